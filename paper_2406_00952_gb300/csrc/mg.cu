// Multigrid preconditioner route for variable a(x) (paper Sec. 3.5, Step 2 by multigrid; Sec. 4).
//
// P_S^{-1} v: time DFT of both halves (zeta = pi scaling, packed as real/imaginary parts), then per
// frequency slot r the 2x2 block G = [[mu_r, -alpha], [alpha, conj(mu_r)]] is decoupled with
// Lemma 3.14 (G = W diag(D1, D2) W^{-1}, W = [[1, M], [M, 1]], D2 = conj(D1)); the two decoupled
// components are solved with `cycles` V-cycles on (D1 I + tau K) -- the second as the conjugate of
// a solve with a conjugated right-hand side -- then recoupled with W and transformed back.
// P_MS^{-1} v (Eq. matrix_P_MS): the same pipeline with no coupling and the real shift
// sigma_r = sqrt(|mu_r|^2 + alpha^2) for both halves.
// Only slots r < n/2 are solved: slot n-1-r carries the conjugate system, whose solution is the
// conjugate (this holds for any real-coefficient linear solver, the V-cycle included, because
// W_{n-1-r} equals conj(W_r) with its columns swapped up to scaling).
//
// V-cycle (reading of an unspecified method): vertex-centred coarsening N -> (N-1)/2, coarse edge
// coefficient = mean of the two fine edges it spans, full-weighting restriction, bilinear
// prolongation, damped Jacobi (weight 4/5), nu1 = nu2 = 2, exact solve on the 1 x 1 grid, zero
// initial guess; cycle c > 1 corrects with a V-cycle on the current residual.
// Neumann grids (Example 3 solved as in Sec. 4, constant a): N = 2^k + 1 nodes per side with the
// boundary, coarse nodes the even fine nodes, N -> (N+1)/2 down to 3; the mirrored stencil
// c (4u - sum of neighbours), c = tau a / h^2, on every level; full weighting with mirrored ghost
// values; bilinear prolongation; the same damped Jacobi; on the 3 x 3 grid an exact solve through
// the eigenvectors of the 3-node mirrored second difference.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "precond_lane.cuh"

namespace pcb {

bool mg_available() { return true; }
int mg_launch_count(int kind);

static constexpr double kJacobiWeight = 0.8;
static constexpr int kMaxLevels = 12;
static constexpr int kNu = 2;
static long long g_mg_launches = 0;   // kernel launches issued by the multigrid route

struct MgLevel {
  int N;                      // interior points per side (Neumann: nodes per side with the boundary)
  int neu;                    // 1: Neumann grid, mirrored stencil with the constant c below
  double c; float cf;         // Neumann: tau a / h^2 of this level
  double* co;                 // Neumann coarsest level: [V2 (81) | V2^{-1} (81) | lambda (9)], FP64 ...
  float* cof;                 // ... and FP32
  double* axs;                // tau/h_l^2 * ax  (N x (N+1))
  double* ays;                // tau/h_l^2 * ay  ((N+1) x N)
  double* dgs;                // sum of the four  (N x N)
  float* axf; float* ayf; float* dgf;
  void* a[3];                 // work arrays: n systems x N^2 complex (FP64-sized)
};

struct MgHost {
  int nlev = 0;
  int nsys = 0;               // systems = n (n/2 frequency slots x 2 right-hand sides)
  int tail_l0 = -1;           // first level of the fused coarse-level launch (-1: none)
  MgLevel lev[kMaxLevels];
  void* zfine = nullptr;      // outer solution (level 0)
  void* xfine = nullptr;      // outer residual (level 0)
  double2* tab_d = nullptr;   // per slot r < n/2: {shift, coupling M, 1/(1-M^2)} for P_S, then P_MS shift
  float2* tab_f = nullptr;
};

// workspace registry: one MgHost per Geom (keyed by the workspace pointer)
static std::vector<std::pair<const void*, MgHost>>& registry() {
  static std::vector<std::pair<const void*, MgHost>> r;
  return r;
}
static MgHost* find_host(const void* ws) {
  for (auto& e : registry())
    if (e.first == ws) return &e.second;
  return nullptr;
}

static int levels_for(int N, bool neu = false) {
  int l = 1;
  if (neu) { while (N > 3) { N = (N + 1) / 2; ++l; } return l; }
  while (N > 1) { N = (N - 1) / 2; ++l; }
  return l;
}

size_t mg_workspace_bytes(const Geom& g) {
  size_t b = 0;
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  int N = g.N;
  const bool neu = g.bc == PCB_BC_NEUMANN;
  const size_t nsys = (size_t)g.n;
  for (int l = 0; l < levels_for(g.N, neu); ++l) {
    const size_t ne = (size_t)N * (N + 1), nn = (size_t)N * N;
    if (!neu) b += up(ne * 8) * 2 + up(nn * 8) + up(ne * 4) * 2 + up(nn * 4);
    b += 3 * up(nsys * nn * sizeof(double2));
    if (l == 0) b += 2 * up(nsys * nn * sizeof(double2));
    N = neu ? (N + 1) / 2 : (N - 1) / 2;
  }
  if (neu) b += up(171 * 8) + up(171 * 4);
  b += up((size_t)g.n * 3 * sizeof(double2)) + up((size_t)g.n * 3 * sizeof(float2));
  return b;
}

// Neumann levels: every level's c = tau a / h_l^2, work arrays, and on the 3 x 3 grid the exact
// solve's tables.  The 3-node mirrored second difference [[2,-2,0],[-1,2,-1],[0,-2,2]] has the
// eigenvalues 0, 2, 4 with eigenvectors (1,1,1), (1,0,-1), (1,-1,1); the 2D operator on the 3 x 3
// grid is c (D (x) I + I (x) D), diagonal in V (x) V.
static unsigned char* mg_setup_neumann(const Geom& g, MgHost& h, unsigned char* p, double a0) {
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  int N = g.N;
  for (int l = 0; l < h.nlev; ++l) {
    MgLevel& L = h.lev[l];
    std::memset(&L, 0, sizeof(L));
    L.N = N; L.neu = 1;
    const double hl = 1.0 / (N - 1);
    L.c = g.tau * a0 / (hl * hl);
    L.cf = (float)L.c;
    const size_t nn = (size_t)N * N;
    for (int k = 0; k < 3; ++k) { L.a[k] = p; p += up((size_t)h.nsys * nn * sizeof(double2)); }
    if (l == 0) {
      h.zfine = p; p += up((size_t)h.nsys * nn * sizeof(double2));
      h.xfine = p; p += up((size_t)h.nsys * nn * sizeof(double2));
    }
    N = (N + 1) / 2;
  }
  MgLevel& C = h.lev[h.nlev - 1];
  const double V[3][3] = {{1, 1, 1}, {1, 0, -1}, {1, -1, 1}};          // columns: eigenvectors
  const double Vi[3][3] = {{0.25, 0.5, 0.25}, {0.5, 0.0, -0.5}, {0.25, -0.5, 0.25}};   // V^{-1}
  const double lam[3] = {0.0, 2.0, 4.0};
  std::vector<double> co(171);
  for (int j = 0; j < 3; ++j)
    for (int i = 0; i < 3; ++i)
      for (int q = 0; q < 3; ++q)
        for (int pp = 0; pp < 3; ++pp) {
          // node (i, j) at 3 j + i, mode (pp, q) at 3 q + pp
          co[(3 * j + i) * 9 + 3 * q + pp] = V[i][pp] * V[j][q];          // V2
          co[81 + (3 * q + pp) * 9 + 3 * j + i] = Vi[pp][i] * Vi[q][j];   // V2^{-1}
        }
  for (int q = 0; q < 3; ++q)
    for (int pp = 0; pp < 3; ++pp) co[162 + 3 * q + pp] = C.c * (lam[pp] + lam[q]);
  std::vector<float> cof(co.begin(), co.end());
  C.co = (double*)p; cudaMemcpy(p, co.data(), 171 * 8, cudaMemcpyHostToDevice); p += up(171 * 8);
  C.cof = (float*)p; cudaMemcpy(p, cof.data(), 171 * 4, cudaMemcpyHostToDevice); p += up(171 * 4);
  return p;
}

static void mg_slot_tables(const Geom& g, MgHost& h, unsigned char*& p);
static int tail_level(const MgHost& h);

cudaError_t mg_setup(Geom& g, void* ws, const double* a_edges, double a0) {
  MgHost h;
  const bool neu = g.bc == PCB_BC_NEUMANN;
  h.nlev = levels_for(g.N, neu);
  if (h.nlev > kMaxLevels) return cudaErrorInvalidValue;
  h.nsys = g.n;
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  unsigned char* p = (unsigned char*)ws;
  if (neu) {
    p = mg_setup_neumann(g, h, p, a0);
    mg_slot_tables(g, h, p);
    h.tail_l0 = tail_level(h);
    if ((size_t)(p - (unsigned char*)ws) > mg_workspace_bytes(g)) return cudaErrorInvalidValue;
    for (auto& e : registry())
      if (e.first == ws) { e.second = h; g.mg = ws; return cudaGetLastError(); }
    registry().push_back({ws, h});
    g.mg = ws;
    return cudaGetLastError();
  }
  // fine coefficients = tau/h^2 * a at the edges; coarser levels average the two fine edges each
  // coarse edge spans and are rescaled with their own spacing
  int N = g.N;
  std::vector<double> ax(a_edges, a_edges + (size_t)N * (N + 1));
  std::vector<double> ay(a_edges + (size_t)N * (N + 1), a_edges + 2 * (size_t)N * (N + 1));
  std::vector<unsigned char> hostbuf;
  for (int l = 0; l < h.nlev; ++l) {
    MgLevel& L = h.lev[l];
    std::memset(&L, 0, sizeof(L));
    L.N = N;
    const double hl = 1.0 / (N + 1), s = g.tau / (hl * hl);
    const size_t ne = (size_t)N * (N + 1), nn = (size_t)N * N;
    std::vector<double> axs(ne), ays(ne), dgs(nn);
    for (size_t k = 0; k < ne; ++k) { axs[k] = s * ax[k]; ays[k] = s * ay[k]; }
    for (int j = 0; j < N; ++j)
      for (int i = 0; i < N; ++i)
        dgs[(size_t)j * N + i] = axs[(size_t)j * (N + 1) + i] + axs[(size_t)j * (N + 1) + i + 1] +
                                 ays[(size_t)j * N + i] + ays[(size_t)(j + 1) * N + i];
    std::vector<float> axf(ne), ayf(ne), dgf(nn);
    for (size_t k = 0; k < ne; ++k) { axf[k] = (float)axs[k]; ayf[k] = (float)ays[k]; }
    for (size_t k = 0; k < nn; ++k) dgf[k] = (float)dgs[k];
    L.axs = (double*)p; cudaMemcpy(p, axs.data(), ne * 8, cudaMemcpyHostToDevice); p += up(ne * 8);
    L.ays = (double*)p; cudaMemcpy(p, ays.data(), ne * 8, cudaMemcpyHostToDevice); p += up(ne * 8);
    L.dgs = (double*)p; cudaMemcpy(p, dgs.data(), nn * 8, cudaMemcpyHostToDevice); p += up(nn * 8);
    L.axf = (float*)p; cudaMemcpy(p, axf.data(), ne * 4, cudaMemcpyHostToDevice); p += up(ne * 4);
    L.ayf = (float*)p; cudaMemcpy(p, ayf.data(), ne * 4, cudaMemcpyHostToDevice); p += up(ne * 4);
    L.dgf = (float*)p; cudaMemcpy(p, dgf.data(), nn * 4, cudaMemcpyHostToDevice); p += up(nn * 4);
    for (int k = 0; k < 3; ++k) { L.a[k] = p; p += up((size_t)h.nsys * nn * sizeof(double2)); }
    if (l == 0) {
      h.zfine = p; p += up((size_t)h.nsys * nn * sizeof(double2));
      h.xfine = p; p += up((size_t)h.nsys * nn * sizeof(double2));
    }
    if (N == 1) break;
    // coarse coefficients: coarse row J sits on fine row 2J+1 (0-based), coarse edge e spans fine
    // edges 2e and 2e+1 (and symmetrically for the x2 edges)
    const int Nc = (N - 1) / 2;
    std::vector<double> axc((size_t)Nc * (Nc + 1)), ayc((size_t)Nc * (Nc + 1));
    for (int J = 0; J < Nc; ++J)
      for (int e = 0; e <= Nc; ++e)
        axc[(size_t)J * (Nc + 1) + e] =
            0.5 * (ax[(size_t)(2 * J + 1) * (N + 1) + 2 * e] + ax[(size_t)(2 * J + 1) * (N + 1) + 2 * e + 1]);
    for (int e = 0; e <= Nc; ++e)
      for (int I = 0; I < Nc; ++I)
        ayc[(size_t)e * Nc + I] = 0.5 * (ay[(size_t)(2 * e) * N + 2 * I + 1] + ay[(size_t)(2 * e + 1) * N + 2 * I + 1]);
    ax.swap(axc); ay.swap(ayc);
    N = Nc;
  }
  mg_slot_tables(g, h, p);
  h.tail_l0 = tail_level(h);
  if ((size_t)(p - (unsigned char*)ws) > mg_workspace_bytes(g)) return cudaErrorInvalidValue;
  for (auto& e : registry())
    if (e.first == ws) { e.second = h; return cudaGetLastError(); }
  registry().push_back({ws, h});
  g.mg = ws;
  return cudaGetLastError();
}

// per-slot table from lambda(S_n) at the F-slots (same formula as the spectral tables)
static void mg_slot_tables(const Geom& g, MgHost& h, unsigned char*& p) {
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const int n = g.n, half = n / 2;
  std::vector<double2> td((size_t)half * 4);
  std::vector<float2> tf((size_t)half * 4);
  for (int r = 0; r < half; ++r) {
    const double psi = -M_PI * (2.0 * r + 1.0) / n;
    const double c = std::cos(psi), s = std::sin(psi);
    const double f1r = 1.0 - c, f1i = -s;
    double f2r = g.theta + (1.0 - g.theta) * c, f2i = (1.0 - g.theta) * s;
    if (std::hypot(f2r, f2i) < 1e-14) { f2r = 1.0; f2i = 0.0; }
    const double den = f2r * f2r + f2i * f2i;
    const double mr = (f1r * f2r + f1i * f2i) / den, mi = (f1i * f2r - f1r * f2i) / den;
    const double a = g.alpha;
    const double sq = std::sqrt(mi * mi + a * a);
    // Lemma 3.14 (principal root): D1 = Re mu + i sqrt(Im^2 mu + alpha^2); M = -(i/alpha)(sq - Im mu)
    const double Mi = -(sq - mi) / a;                 // M = i * Mi (purely imaginary)
    const double inv = 1.0 / (1.0 + Mi * Mi);         // 1/(1 - M^2) with M^2 = -Mi^2
    td[4 * r + 0] = make_double2(mr, sq);             // D1
    td[4 * r + 1] = make_double2(0.0, Mi);            // M
    td[4 * r + 2] = make_double2(inv, 0.0);
    td[4 * r + 3] = make_double2(std::sqrt(mr * mr + mi * mi + a * a), 0.0);   // P_MS shift sigma_r
    for (int k = 0; k < 4; ++k) tf[4 * r + k] = make_float2((float)td[4 * r + k].x, (float)td[4 * r + k].y);
  }
  h.tab_d = (double2*)p; cudaMemcpy(p, td.data(), td.size() * sizeof(double2), cudaMemcpyHostToDevice);
  p += up(td.size() * sizeof(double2));
  h.tab_f = (float2*)p; cudaMemcpy(p, tf.data(), tf.size() * sizeof(float2), cudaMemcpyHostToDevice);
  p += up(tf.size() * sizeof(float2));
}

void mg_release(const void* ws) {
  auto& r = registry();
  for (size_t k = 0; k < r.size(); ++k)
    if (r[k].first == ws) { r.erase(r.begin() + k); return; }
}

// ------------------------------------------------------------------------------------------
// kernels (one instance; thread per (system, grid point)).  Blocks of 32 x 8 threads cover tiles
// of 32 x 8 points of one system's grid (grid x, y over the tiles, z over the systems), so that
// consecutive threads touch consecutive points and no index needs a division.
// ------------------------------------------------------------------------------------------
struct GridPt { int b, i, j; };
__device__ __forceinline__ GridPt grid_pt() {
  return GridPt{(int)blockIdx.z, (int)(blockIdx.x * 32 + threadIdx.x), (int)(blockIdx.y * 8 + threadIdx.y)};
}
static dim3 grid_for(int N, int nsys) { return dim3((unsigned)((N + 31) / 32), (unsigned)((N + 7) / 8), (unsigned)nsys); }
static const dim3 kMgBlock(32, 8);
template <typename R> struct Coef;
template <> struct Coef<float> {
  static __device__ const float* ax(const MgLevel& L) { return L.axf; }
  static __device__ const float* ay(const MgLevel& L) { return L.ayf; }
  static __device__ const float* dg(const MgLevel& L) { return L.dgf; }
};
template <> struct Coef<double> {
  static __device__ const double* ax(const MgLevel& L) { return L.axs; }
  static __device__ const double* ay(const MgLevel& L) { return L.ays; }
  static __device__ const double* dg(const MgLevel& L) { return L.dgs; }
};

// (tau K z) at point (i, j) of system b
template <typename R>
__device__ __forceinline__ cx<R> tauKz(const MgLevel& L, const cx<R>* __restrict__ z, int i, int j) {
  const int N = L.N;
  if (L.neu) {   // mirrored neighbours: u_{-1} = u_1, u_N = u_{N-2}
    const R c = sizeof(R) == 4 ? (R)L.cf : (R)L.c;
    const cx<R> l = z[j * N + (i > 0 ? i - 1 : 1)], r = z[j * N + (i < N - 1 ? i + 1 : N - 2)];
    const cx<R> d = z[(j > 0 ? j - 1 : 1) * N + i], t = z[(j < N - 1 ? j + 1 : N - 2) * N + i];
    const cx<R> nb = cadd(cadd(l, r), cadd(d, t));
    return cscale(csub(cscale(z[j * N + i], (R)4), nb), c);
  }
  const R* ax = Coef<R>::ax(L) + (long long)j * (N + 1);
  const R* ay = Coef<R>::ay(L);
  const cx<R> c = z[j * N + i];
  cx<R> s = mk<R>(0, 0);
  if (i > 0) s = cadd(s, cscale(z[j * N + i - 1], ax[i]));
  if (i < N - 1) s = cadd(s, cscale(z[j * N + i + 1], ax[i + 1]));
  if (j > 0) s = cadd(s, cscale(z[(j - 1) * N + i], ay[(long long)j * N + i]));
  if (j < N - 1) s = cadd(s, cscale(z[(j + 1) * N + i], ay[(long long)(j + 1) * N + i]));
  const R d = Coef<R>::dg(L)[j * N + i];
  return csub(cscale(c, d), s);
}

template <typename R>
__device__ __forceinline__ cx<R> shift_of(const cx<R>* __restrict__ tab, int b, int kind) {
  const int r = b >> 1;
  return kind == 2 ? tab[4 * r + 0] : mk<R>(tab[4 * r + 3].x, (R)0);
}

// Per-point operations, shared by the one-launch-per-step kernels of the fine levels and the
// fused kernel of the coarse levels (identical arithmetic on either path).  Arrays hold one
// system's grid, row j of N points at j N.

// Jacobi diagonal inverse of system shift mu at point pt
template <typename R>
__device__ __forceinline__ cx<R> jacobi_dinv(const MgLevel& L, cx<R> mu, int pt) {
  const R dgk = L.neu ? (R)4 * (sizeof(R) == 4 ? (R)L.cf : (R)L.c) : Coef<R>::dg(L)[pt];
  const cx<R> d = mk<R>(mu.x + dgk, mu.y);
  const R rd = (R)1 / (d.x * d.x + d.y * d.y);
  return mk<R>(d.x * rd, -d.y * rd);
}

// one damped Jacobi update at (i, j): out = z + w (rhs - A z) / diag (first: z = 0)
template <typename R>
__device__ __forceinline__ cx<R> jacobi_pt(const MgLevel& L, cx<R> mu, cx<R> dinv, const cx<R>* __restrict__ rhs,
                                           const cx<R>* __restrict__ z, int i, int j, bool first, R w) {
  const int pt = j * L.N + i;
  if (first) return cscale(cmul(rhs[pt], dinv), w);
  const cx<R> Az = cadd(cmul(mu, z[pt]), tauKz<R>(L, z, i, j));
  return cadd(z[pt], cscale(cmul(csub(rhs[pt], Az), dinv), w));
}

// residual rhs - A z at (i, j)
template <typename R>
__device__ __forceinline__ cx<R> resid_pt(const MgLevel& L, cx<R> mu, const cx<R>* __restrict__ rhs,
                                          const cx<R>* __restrict__ z, int i, int j) {
  const int pt = j * L.N + i;
  const cx<R> Az = cadd(cmul(mu, z[pt]), tauKz<R>(L, z, i, j));
  return csub(rhs[pt], Az);
}

// full weighting: coarse (I, J) <- fine 9-point neighbourhood of (2I+1, 2J+1) (0-based); Neumann:
// of (2I, 2J) with mirrored ghost values
template <typename R>
__device__ __forceinline__ cx<R> restrict_pt(int Nf, bool neu, const cx<R>* fb, int I, int J) {
  const int fi = neu ? 2 * I : 2 * I + 1, fj = neu ? 2 * J : 2 * J + 1;
  auto mir = [&](int k) { return k < 0 ? -k : (k > Nf - 1 ? 2 * (Nf - 1) - k : k); };
  auto at = [&](int ii, int jj) { return neu ? fb[mir(jj) * Nf + mir(ii)] : fb[jj * Nf + ii]; };
  cx<R> s = cscale(at(fi, fj), (R)4);
  s = cadd(s, cscale(cadd(cadd(at(fi - 1, fj), at(fi + 1, fj)), cadd(at(fi, fj - 1), at(fi, fj + 1))), (R)2));
  s = cadd(s, cadd(cadd(at(fi - 1, fj - 1), at(fi + 1, fj - 1)), cadd(at(fi - 1, fj + 1), at(fi + 1, fj + 1))));
  return cscale(s, (R)(1.0 / 16.0));
}

// bilinear prolongation of the coarse grid cb (Nc points per side) at fine (i, j).  Dirichlet:
// fine 0-based index 2K+1 sits on coarse node K, an even fine index between nodes K-1 and K; with
// Ka = (k-1) >> 1 and Kb = k >> 1 in each direction (equal for an odd k) the value is 1/4 of the
// sum over the four (Ka|Kb) pairs, which equals the one-, two- or four-node average exactly
// (scalings by powers of two), so no thread branches on the parity of its point.  Neumann: even
// fine nodes are coarse nodes.
template <typename R>
__device__ __forceinline__ cx<R> prolong_pt(int Nc, bool neu, const cx<R>* cb, int i, int j) {
  if (neu) {
    const int I0 = i >> 1, J0 = j >> 1, I1 = (i + 1) >> 1, J1 = (j + 1) >> 1;   // equal when even
    return cscale(cadd(cadd(cb[J0 * Nc + I0], cb[J0 * Nc + I1]), cadd(cb[J1 * Nc + I0], cb[J1 * Nc + I1])), (R)0.25);
  }
  const int Ia = (i - 1) >> 1, Ib = i >> 1, Ja = (j - 1) >> 1, Jb = j >> 1;
  const bool xa = Ia >= 0, xb = Ib < Nc, ya = Ja >= 0, yb = Jb < Nc;
  const cx<R> zero = mk<R>(0, 0);
  const cx<R> c11 = xa && ya ? cb[Ja * Nc + Ia] : zero, c21 = xb && ya ? cb[Ja * Nc + Ib] : zero;
  const cx<R> c12 = xa && yb ? cb[Jb * Nc + Ia] : zero, c22 = xb && yb ? cb[Jb * Nc + Ib] : zero;
  return cscale(cadd(cadd(c11, c21), cadd(c12, c22)), (R)0.25);
}

// Neumann 3 x 3 grid: exact solve z = V2 diag(1/(mu + lambda)) V2^{-1} rhs at `node`
template <typename R>
__device__ __forceinline__ cx<R> coarse_neu_pt(const MgLevel& L, cx<R> mu, const cx<R>* rb, int node) {
  const R* co = sizeof(R) == 4 ? (const R*)L.cof : (const R*)L.co;
  cx<R> acc = mk<R>(0, 0);
  for (int md = 0; md < 9; ++md) {
    cx<R> w = mk<R>(0, 0);
    for (int k = 0; k < 9; ++k) w = cadd(w, cscale(rb[k], co[81 + md * 9 + k]));
    const cx<R> den = mk<R>(mu.x + co[162 + md], mu.y);
    const R dd = den.x * den.x + den.y * den.y;
    w = cmul(w, mk<R>(den.x / dd, -den.y / dd));
    acc = cadd(acc, cscale(w, co[node * 9 + md]));
  }
  return acc;
}

// The two systems of a frequency slot (2r and 2r + 1) share the shift and hence the diagonal:
// a thread treats one grid point of both (grid z runs over the slots).

template <typename R, bool FIRST>
__global__ void __launch_bounds__(256) k_mg_jacobi(MgLevel L, const cx<R>* __restrict__ tab, int kind,
                                                   const cx<R>* __restrict__ rhs, const cx<R>* __restrict__ z,
                                                   cx<R>* __restrict__ out, R w) {
  const int N = L.N, nn = N * N;
  const GridPt q = grid_pt();
  if (q.i >= N || q.j >= N) return;
  const int b = 2 * q.b, pt = q.j * N + q.i;
  const cx<R> mu = shift_of<R>(tab, b, kind);
  const cx<R> dinv = jacobi_dinv<R>(L, mu, pt);
  const long long o0 = (long long)b * nn, o1 = o0 + nn;
  if (FIRST) {
    const cx<R> r0 = rhs[o0 + pt], r1 = rhs[o1 + pt];
    out[o0 + pt] = cscale(cmul(r0, dinv), w);
    out[o1 + pt] = cscale(cmul(r1, dinv), w);
    return;
  }
  // jacobi_pt's arithmetic, with both systems' products formed before either update so that all
  // loads are in flight together
  const cx<R> Az0 = cadd(cmul(mu, z[o0 + pt]), tauKz<R>(L, z + o0, q.i, q.j));
  const cx<R> Az1 = cadd(cmul(mu, z[o1 + pt]), tauKz<R>(L, z + o1, q.i, q.j));
  const cx<R> n0 = cadd(z[o0 + pt], cscale(cmul(csub(rhs[o0 + pt], Az0), dinv), w));
  const cx<R> n1 = cadd(z[o1 + pt], cscale(cmul(csub(rhs[o1 + pt], Az1), dinv), w));
  out[o0 + pt] = n0;
  out[o1 + pt] = n1;
}

template <typename R>
__global__ void __launch_bounds__(256) k_mg_resid(MgLevel L, const cx<R>* __restrict__ tab, int kind,
                                                  const cx<R>* __restrict__ rhs, const cx<R>* __restrict__ z,
                                                  cx<R>* __restrict__ res) {
  const int N = L.N, nn = N * N;
  const GridPt q = grid_pt();
  if (q.i >= N || q.j >= N) return;
  const int b = 2 * q.b, pt = q.j * N + q.i;
  const cx<R> mu = shift_of<R>(tab, b, kind);
  const long long o0 = (long long)b * nn, o1 = o0 + nn;
  const cx<R> r0 = resid_pt<R>(L, mu, rhs + o0, z + o0, q.i, q.j);
  const cx<R> r1 = resid_pt<R>(L, mu, rhs + o1, z + o1, q.i, q.j);
  res[o0 + pt] = r0;
  res[o1 + pt] = r1;
}

// The fused smoothing of a Dirichlet level.  A block takes a 32 x 16 tile of both systems of a slot, with
// the two systems' values side by side (one 16-byte access for both).  Every point's stencil coefficients
// and Jacobi weight are formed once for both systems and the weight once for both sweeps: with 32 x 8
// tiles, a weight per sweep and separate systems, instructions bound the pre-smoothing (level 0 at N = 255,
// n = 256: 181 us, now 136; its traffic alone takes 59 us).
template <typename R> struct alignas(4 * sizeof(R)) Duo { cx<R> v[2]; };
namespace tile {
constexpr int TX = 32, TY = 16, WX2 = TX + 4, WY2 = TY + 4, WX1 = TX + 2, WY1 = TY + 2;
}
static dim3 tile_grid(int N, int nslot) {
  return dim3((unsigned)((N + tile::TX - 1) / tile::TX), (unsigned)((N + tile::TY - 1) / tile::TY), (unsigned)nslot);
}

// (mu I + tau K) z at grid point (gi, gj) from a window of row pitch WX whose entry (gi, gj) is zs[at], for both
// systems: the arithmetic of tauKz.  The window holds zeros outside the grid.
template <typename R, int WX>
__device__ __forceinline__ Duo<R> shifted_win(const MgLevel& L, cx<R> mu, const Duo<R>* zs, int at, int gi, int gj) {
  const int N = L.N, pt = gj * N + gi;
  const R* ax = Coef<R>::ax(L) + pt + gj;              // rows of N + 1 edges
  const R* ay = Coef<R>::ay(L) + pt;
  const R al = __ldg(ax), ar = __ldg(ax + 1), ad = __ldg(ay), au = __ldg(ay + N), d = __ldg(Coef<R>::dg(L) + pt);
  const Duo<R> c = zs[at], l = zs[at - 1], r = zs[at + 1], dn = zs[at - WX], up = zs[at + WX];
  Duo<R> o;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    cx<R> s = cscale(l.v[k], al);
    s = cadd(s, cscale(r.v[k], ar));
    s = cadd(s, cscale(dn.v[k], ad));
    s = cadd(s, cscale(up.v[k], au));
    o.v[k] = cadd(cmul(mu, c.v[k]), csub(cscale(c.v[k], d), s));
  }
  return o;
}
// one damped Jacobi update from the window
template <typename R, int WX>
__device__ __forceinline__ Duo<R> jacobi_win(const MgLevel& L, cx<R> mu, cx<R> dinv, const Duo<R>& r, const Duo<R>* zs,
                                             int at, int gi, int gj, R w) {
  const Duo<R> Az = shifted_win<R, WX>(L, mu, zs, at, gi, gj), c = zs[at];
  Duo<R> o;
#pragma unroll
  for (int k = 0; k < 2; ++k) o.v[k] = cadd(c.v[k], cscale(cmul(csub(r.v[k], Az.v[k]), dinv), w));
  return o;
}

// The pre-smoothing (two sweeps, the first from zero) and the residual of its result: the right-hand sides
// on the tile with a halo of two points, the first sweep there, the second with a halo of one, and the
// residual on the tile.  Reads one grid and writes two, where the separate launches moved eight.
template <typename R>
__global__ void __launch_bounds__(256) k_mg_presmooth(MgLevel L, const cx<R>* __restrict__ tab, int kind,
                                                      const cx<R>* __restrict__ rhs, cx<R>* __restrict__ zout,
                                                      cx<R>* __restrict__ res, R w) {
  using C = cx<R>;
  using namespace tile;
  __shared__ Duo<R> r2[WX2 * WY2], z1[WX2 * WY2], z2[WX1 * WY1];
  __shared__ C di[WX2 * WY2];
  const int N = L.N, nn = N * N;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, tid = threadIdx.y * TX + threadIdx.x;
  const C mu = shift_of<R>(tab, 2 * blockIdx.z, kind);
  const long long o0 = 2LL * blockIdx.z * nn, o1 = o0 + nn;
  const C zero = mk<R>(0, 0);
  for (int e = tid; e < WX2 * WY2; e += 256) {
    const int lj = e / WX2, li = e - lj * WX2, gi = x0 - 2 + li, gj = y0 - 2 + lj;
    Duo<R> r{{zero, zero}}, z{{zero, zero}};
    C dinv = zero;
    if (gi >= 0 && gi < N && gj >= 0 && gj < N) {
      const int pt = gj * N + gi;
      r.v[0] = rhs[o0 + pt];
      r.v[1] = rhs[o1 + pt];
      dinv = jacobi_dinv<R>(L, mu, pt);
#pragma unroll
      for (int k = 0; k < 2; ++k) z.v[k] = cscale(cmul(r.v[k], dinv), w);
    }
    r2[e] = r;
    z1[e] = z;
    di[e] = dinv;
  }
  __syncthreads();
  for (int e = tid; e < WX1 * WY1; e += 256) {
    const int lj = e / WX1, li = e - lj * WX1, gi = x0 - 1 + li, gj = y0 - 1 + lj, at = (lj + 1) * WX2 + li + 1;
    Duo<R> z{{zero, zero}};
    if (gi >= 0 && gi < N && gj >= 0 && gj < N) z = jacobi_win<R, WX2>(L, mu, di[at], r2[at], z1, at, gi, gj, w);
    z2[e] = z;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int ty = threadIdx.y + 8 * h, gi = x0 + threadIdx.x, gj = y0 + ty;
    if (gi < N && gj < N) {
      const int at = (ty + 1) * WX1 + threadIdx.x + 1, pt = gj * N + gi;
      const Duo<R> Az = shifted_win<R, WX1>(L, mu, z2, at, gi, gj), zc = z2[at];
      const Duo<R> r = r2[(ty + 2) * WX2 + threadIdx.x + 2];
      zout[o0 + pt] = zc.v[0];
      zout[o1 + pt] = zc.v[1];
      res[o0 + pt] = csub(r.v[0], Az.v[0]);
      res[o1 + pt] = csub(r.v[1], Az.v[1]);
    }
  }
}

// The coarse correction and the two post-smoothing sweeps: z plus the prolonged correction on the tile with
// a halo of two points, one sweep with a halo of one, the second on the tile.  Reads two grids and a
// quarter and writes one, where the separate launches moved eight and a quarter (level 0 at N = 255,
// n = 256: 48 + 2 x 93 us, now 180; its traffic alone takes 64).  `base` (a further cycle, whose z corrects
// base): the result is added there and not written to zout.
template <typename R>
__global__ void __launch_bounds__(256) k_mg_postsmooth(MgLevel L, const cx<R>* __restrict__ tab, int kind,
                                                       const cx<R>* __restrict__ rhs, const cx<R>* __restrict__ zin,
                                                       const cx<R>* __restrict__ coarse, cx<R>* __restrict__ zout,
                                                       cx<R>* __restrict__ base, R w) {
  using C = cx<R>;
  using namespace tile;
  constexpr int CX = TX / 2 + 3, CY = TY / 2 + 3;      // coarse points -2 .. TX/2 of the tile's corner
  __shared__ Duo<R> cw[CX * CY], z0[WX2 * WY2], r1[WX1 * WY1], z1[WX1 * WY1];
  __shared__ C di[WX1 * WY1];
  const int N = L.N, nn = N * N, Nc = (N - 1) / 2, nnc = Nc * Nc;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, tid = threadIdx.y * TX + threadIdx.x;
  const C mu = shift_of<R>(tab, 2 * blockIdx.z, kind);
  const long long o0 = 2LL * blockIdx.z * nn, o1 = o0 + nn;
  const C* __restrict__ c0 = coarse + 2LL * blockIdx.z * nnc;
  const C zero = mk<R>(0, 0);
  for (int e = tid; e < CX * CY; e += 256) {
    const int lj = e / CX, ci = x0 / 2 - 2 + e - lj * CX, cj = y0 / 2 - 2 + lj;
    const bool in = ci >= 0 && ci < Nc && cj >= 0 && cj < Nc;
    cw[e].v[0] = in ? c0[cj * Nc + ci] : zero;
    cw[e].v[1] = in ? c0[nnc + cj * Nc + ci] : zero;
  }
  __syncthreads();
  for (int e = tid; e < WX2 * WY2; e += 256) {
    const int lj = e / WX2, li = e - lj * WX2, gi = x0 - 2 + li, gj = y0 - 2 + lj;
    Duo<R> z{{zero, zero}};
    if (gi >= 0 && gi < N && gj >= 0 && gj < N) {
      const int pt = gj * N + gi;
      // prolong_pt's sum over (Ka|Kb) pairs, from the window
      const int ia = (li + 1) >> 1, ib = (li + 2) >> 1, ja = ((lj + 1) >> 1) * CX, jb = ((lj + 2) >> 1) * CX;
      const Duo<R> c11 = cw[ja + ia], c21 = cw[ja + ib], c12 = cw[jb + ia], c22 = cw[jb + ib];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        z.v[k] = cadd(zin[(k ? o1 : o0) + pt],
                      cscale(cadd(cadd(c11.v[k], c21.v[k]), cadd(c12.v[k], c22.v[k])), (R)0.25));
    }
    z0[e] = z;
  }
  __syncthreads();
  for (int e = tid; e < WX1 * WY1; e += 256) {
    const int lj = e / WX1, li = e - lj * WX1, gi = x0 - 1 + li, gj = y0 - 1 + lj, at = (lj + 1) * WX2 + li + 1;
    Duo<R> r{{zero, zero}}, z{{zero, zero}};
    C dinv = zero;
    if (gi >= 0 && gi < N && gj >= 0 && gj < N) {
      const int pt = gj * N + gi;
      r.v[0] = rhs[o0 + pt];
      r.v[1] = rhs[o1 + pt];
      dinv = jacobi_dinv<R>(L, mu, pt);
      z = jacobi_win<R, WX2>(L, mu, dinv, r, z0, at, gi, gj, w);
    }
    r1[e] = r;
    di[e] = dinv;
    z1[e] = z;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int ty = threadIdx.y + 8 * h, gi = x0 + threadIdx.x, gj = y0 + ty;
    if (gi < N && gj < N) {
      const int at = (ty + 1) * WX1 + threadIdx.x + 1, pt = gj * N + gi;
      const Duo<R> z = jacobi_win<R, WX1>(L, mu, di[at], r1[at], z1, at, gi, gj, w);
      if (base) {
        base[o0 + pt] = cadd(base[o0 + pt], z.v[0]);
        base[o1 + pt] = cadd(base[o1 + pt], z.v[1]);
      } else {
        zout[o0 + pt] = z.v[0];
        zout[o1 + pt] = z.v[1];
      }
    }
  }
}

template <typename R, bool NEU>
__global__ void __launch_bounds__(256) k_mg_restrict(int Nf, const cx<R>* __restrict__ f, cx<R>* __restrict__ c) {
  const int Nc = NEU ? (Nf + 1) / 2 : (Nf - 1) / 2, nnc = Nc * Nc, nnf = Nf * Nf;
  const GridPt q = grid_pt();
  if (q.i >= Nc || q.j >= Nc) return;
  const cx<R> v0 = restrict_pt<R>(Nf, NEU, f + 2LL * q.b * nnf, q.i, q.j);
  const cx<R> v1 = restrict_pt<R>(Nf, NEU, f + (2LL * q.b + 1) * nnf, q.i, q.j);
  c[2LL * q.b * nnc + q.j * Nc + q.i] = v0;
  c[(2LL * q.b + 1) * nnc + q.j * Nc + q.i] = v1;
}

// the prolonged coarse correction added to the fine solution
template <typename R, bool NEU>
__global__ void __launch_bounds__(256) k_mg_prolong_add(int Nf, const cx<R>* __restrict__ c, cx<R>* __restrict__ z) {
  const int Nc = NEU ? (Nf + 1) / 2 : (Nf - 1) / 2, nnc = Nc * Nc, nnf = Nf * Nf;
  const GridPt q = grid_pt();
  if (q.i >= Nf || q.j >= Nf) return;
  const long long o0 = 2LL * q.b * nnf + q.j * Nf + q.i, o1 = o0 + nnf;
  const cx<R> v0 = prolong_pt<R>(Nc, NEU, c + 2LL * q.b * nnc, q.i, q.j);
  const cx<R> v1 = prolong_pt<R>(Nc, NEU, c + (2LL * q.b + 1) * nnc, q.i, q.j);
  const cx<R> z0 = z[o0], z1 = z[o1];
  z[o0] = cadd(z0, v0);
  z[o1] = cadd(z1, v1);
}

// Neumann 3 x 3 grid, one thread per (system, node)
template <typename R>
__global__ void k_mg_coarse_neu(MgLevel L, int nsys, const cx<R>* __restrict__ tab, int kind,
                                const cx<R>* __restrict__ rhs, cx<R>* __restrict__ z) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)nsys * 9) return;
  const int b = (int)(idx / 9), node = (int)(idx - (long long)b * 9);
  z[(long long)b * 9 + node] = coarse_neu_pt<R>(L, shift_of<R>(tab, b, kind), rhs + (long long)b * 9, node);
}

// ------------------------------------------------------------------------------------------
// The coarse levels in one launch.  Below about 33 points per side a level's steps are too small
// to fill the GPU, and each one-per-step launch costs several microseconds whatever its size.
// One block takes both systems of a slot through the V-cycle from level l0 down to the coarsest
// grid and back, with every level's right-hand side, solution and spare grid in shared memory,
// the same per-point arithmetic as the fine levels, and a block barrier between steps.
// ------------------------------------------------------------------------------------------
struct MgTail {
  MgLevel lev[kMaxLevels];
  int l0, nlev;
};

template <typename R>
size_t tail_smem(const MgTail& t) {
  size_t e = 0;
  for (int l = t.l0; l < t.nlev; ++l) e += 3 * 2 * (size_t)t.lev[l].N * t.lev[l].N;
  return e * sizeof(cx<R>);
}

static constexpr size_t kTailSmemMax = 200 * 1024;
static_assert(kNu % 2 == 0, "the fused coarse levels expect the pre-smoothing to end in z");

// first level of the fused launch: the first below the finest with at most 33 points per side whose
// levels fit the shared-memory budget in FP64; -1 if none
static int tail_level(const MgHost& h) {
  for (int l = 1; l < h.nlev; ++l) {
    if (h.lev[l].N > 33) continue;
    MgTail T;
    for (int k = 0; k < h.nlev; ++k) T.lev[k] = h.lev[k];
    T.l0 = l; T.nlev = h.nlev;
    return tail_smem<double>(T) <= kTailSmemMax ? l : -1;
  }
  return -1;
}

template <typename R>
__global__ void __launch_bounds__(256) k_mg_vcycle_tail(MgTail T, const cx<R>* __restrict__ tab, int kind,
                                                        const cx<R>* __restrict__ grhs, cx<R>* __restrict__ gz) {
  using C = cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* base[kMaxLevels][3];                         // [level][rhs, z, spare], each 2 systems x N^2
  {
    C* p = (C*)smem_raw;
    for (int l = T.l0; l < T.nlev; ++l) {
      const int nn2 = 2 * T.lev[l].N * T.lev[l].N;
      for (int a = 0; a < 3; ++a) { base[l][a] = p; p += nn2; }
    }
  }
  const int slot = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const cx<R> mu = shift_of<R>(tab, 2 * slot, kind);
  const R w = (R)kJacobiWeight;
  {   // right-hand sides of level l0
    const int nn = T.lev[T.l0].N * T.lev[T.l0].N;
    const C* src = grhs + (long long)2 * slot * nn;
    for (int e = tid; e < 2 * nn; e += nt) base[T.l0][0][e] = src[e];
  }
  __syncthreads();
  // sweep over every (system, point) of level l
  auto each = [&](int l, auto&& f) {
    const int N = T.lev[l].N, nn = N * N;
    for (int e = tid; e < 2 * nn; e += nt) {
      const int k = e >= nn ? 1 : 0, pt = e - k * nn, j = pt / N, i = pt - j * N;
      f(k, pt, i, j, nn);
    }
    __syncthreads();
  };
  // descent: nu1 sweeps (the first from zero, into `spare`, so that the last post-smoothing
  // sweep lands in z), residual, restriction
  for (int l = T.l0; l < T.nlev - 1; ++l) {
    const MgLevel& L = T.lev[l];
    C* rhs = base[l][0];
    C* cur = base[l][2];
    C* oth = base[l][1];
    each(l, [&](int k, int pt, int i, int j, int nn) {
      cur[k * nn + pt] = jacobi_pt<R>(L, mu, jacobi_dinv<R>(L, mu, pt), rhs + k * nn, nullptr, i, j, true, w);
    });
    for (int s = 1; s < kNu; ++s) {
      each(l, [&](int k, int pt, int i, int j, int nn) {
        oth[k * nn + pt] = jacobi_pt<R>(L, mu, jacobi_dinv<R>(L, mu, pt), rhs + k * nn, cur + k * nn, i, j, false, w);
      });
      C* t = cur; cur = oth; oth = t;
    }
    each(l, [&](int k, int pt, int i, int j, int nn) {
      oth[k * nn + pt] = resid_pt<R>(L, mu, rhs + k * nn, cur + k * nn, i, j);
    });
    each(l + 1, [&](int k, int pt, int i, int j, int nn) {
      base[l + 1][0][k * nn + pt] = restrict_pt<R>(L.N, L.neu != 0, oth + k * L.N * L.N, i, j);
    });
  }
  {   // coarsest grid: exact solve
    const int l = T.nlev - 1;
    const MgLevel& L = T.lev[l];
    C* rhs = base[l][0];
    C* z = base[l][1];
    each(l, [&](int k, int pt, int i, int j, int nn) {
      z[k * nn + pt] = L.neu ? coarse_neu_pt<R>(L, mu, rhs + k * nn, pt)
                             : jacobi_pt<R>(L, mu, jacobi_dinv<R>(L, mu, pt), rhs + k * nn, nullptr, i, j, true, (R)1);
    });
  }
  // ascent: prolongation added into z, nu2 sweeps ending in z
  for (int l = T.nlev - 2; l >= T.l0; --l) {
    const MgLevel& L = T.lev[l];
    const int Nc = T.lev[l + 1].N;
    C* rhs = base[l][0];
    C* cur = base[l][1];
    C* oth = base[l][2];
    each(l, [&](int k, int pt, int i, int j, int nn) {
      cur[k * nn + pt] = cadd(cur[k * nn + pt], prolong_pt<R>(Nc, L.neu != 0, base[l + 1][1] + k * Nc * Nc, i, j));
    });
    for (int s = 0; s < kNu; ++s) {
      each(l, [&](int k, int pt, int i, int j, int nn) {
        oth[k * nn + pt] = jacobi_pt<R>(L, mu, jacobi_dinv<R>(L, mu, pt), rhs + k * nn, cur + k * nn, i, j, false, w);
      });
      C* t = cur; cur = oth; oth = t;
    }
  }
  {   // solution of level l0
    const int nn = T.lev[T.l0].N * T.lev[T.l0].N;
    C* dst = gz + (long long)2 * slot * nn;
    for (int e = tid; e < 2 * nn; e += nt) dst[e] = base[T.l0][1][e];
  }
}

// a += b  or  a = b (copy)
template <typename R>
__global__ void k_mg_axpy(long long len, const cx<R>* __restrict__ src, cx<R>* __restrict__ dst, int copy) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= len) return;
  dst[idx] = copy ? src[idx] : cadd(dst[idx], src[idx]);
}

// ------------------------------------------------------------------------------------------
// time passes around the multigrid
// ------------------------------------------------------------------------------------------
// The transforms of precond_lane.cuh (n = A B, two register steps with one exchange) with one column per
// lane: the forward pass ends in the decoupled right-hand sides, the inverse one begins with the
// recoupling.  A slot pair (r, n-1-r) is held by one thread, so the coupling needs no second exchange, and
// every global access of a half warp is a full 128-byte line.  Both are bound by HBM and by the
// conversions between FP64 and FP32, half of which go to the integer pipe (f32_convert.cuh).  The kernels
// before them gave a column to a warp and wrote the slots of one column side by side, m values apart:
// N = 255, n = 256, FP32 197 + 172 us, now 88 + 90 us (the traffic alone takes 59 us each).
template <typename R, int n>
constexpr int mg_time_columns() { return lane::TimeShape<R, n>::B == 1 ? 128 : lane::time_lanes<R, n, false>(); }
template <typename R, int n>
constexpr int mg_time_threads() { return lane::TimeShape<R, n>::B == 1 ? 128 : lane::time_threads<R, n, false>(); }

// x[q] = the pair of halves at p[q step] in R, q < A
template <typename R, int A>
__device__ __forceinline__ void load_pairs(cx<R>* x, const double* __restrict__ p, const double* __restrict__ p2,
                                           long long step) {
  if constexpr (sizeof(R) == 8) {
#pragma unroll
    for (int q = 0; q < A; ++q) x[q] = mk<R>(p[q * step], p2[q * step]);
  } else {
    unsigned rare = 0;
#pragma unroll
    for (int q = 0; q < A; ++q) x[q] = mk<R>((R)p[q * step], (R)d2f_plain(p2[q * step], rare));
    if (rare) {
#pragma unroll
      for (int q = 0; q < A; ++q) x[q].y = (R)p2[q * step];
    }
  }
}
template <typename R>
__device__ __forceinline__ void store_pair(double* p, double* p2, cx<R> v, unsigned& rare) {
  *p = (double)v.x;
  if constexpr (sizeof(R) == 8) *p2 = v.y;
  else *p2 = f2d_plain(v.y, rare);
}

// right-hand sides of slot r (systems 2r and 2r + 1) from C_r and C_{n-1-r}
template <typename R>
__device__ __forceinline__ void put_slot(cx<R>* __restrict__ rhs, const cx<R>* __restrict__ tab, int kind, long long m,
                                         int r, cx<R> Cr, cx<R> Cq) {
  using T = cx<R>;
  Cq = cconj(Cq);
  const T F1 = cscale(cadd(Cr, Cq), (R)0.5);
  const T F2 = cmul_mi(cscale(csub(Cr, Cq), (R)0.5));
  T T1 = F1, T2 = F2;
  if (kind == 2) {   // W^{-1} [F1; F2], W = [[1, M], [M, 1]]
    const T M = __ldg(&tab[4 * r + 1]);
    const R inv = __ldg(&tab[4 * r + 2]).x;
    T1 = cscale(csub(F1, cmul(M, F2)), inv);
    T2 = cscale(csub(F2, cmul(M, F1)), inv);
    T2 = cconj(T2);   // second component: solved as the conjugate system with D1
  }
  rhs[2 * r * m] = T1;
  rhs[(2 * r + 1) * m] = T2;
}
// C_r and C_{n-1-r} from the solutions of slot r
template <typename R>
__device__ __forceinline__ void get_slot(const cx<R>* __restrict__ z, const cx<R>* __restrict__ tab, int kind,
                                         long long m, int r, cx<R>& Cr, cx<R>& Cq) {
  using T = cx<R>;
  const T Z1 = z[2 * r * m];
  T Z2 = z[(2 * r + 1) * m];
  T U1 = Z1, U2 = Z2;
  if (kind == 2) {
    Z2 = cconj(Z2);
    const T M = __ldg(&tab[4 * r + 1]);
    U1 = cadd(Z1, cmul(M, Z2));
    U2 = cadd(cmul(M, Z1), Z2);
  }
  Cr = cadd(U1, cmul_pi(U2));
  Cq = cadd(cconj(U1), cmul_pi(cconj(U2)));
}

// forward: v (FP64, 2 halves) -> right-hand sides of the n systems (slot r < n/2: 2r and 2r+1)
template <typename R, int n>
__global__ void __launch_bounds__((mg_time_threads<R, n>()), (lane::time_blocks_per_sm<R, n, false>()))
    k_mg_time_fwd(const Geom* __restrict__ G, const Slots* __restrict__ S, int in_slot, const cx<R>* __restrict__ tab,
                  int kind, cx<R>* __restrict__ rhs) {
  using T = cx<R>;
  constexpr int A = lane::TimeShape<R, n>::A, B = lane::TimeShape<R, n>::B;
  constexpr int LT = mg_time_columns<R, n>(), NG = mg_time_threads<R, n>() / LT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geom& g = G[0];
  const int m = g.m, l = threadIdx.x % LT, grp = threadIdx.x / LT;
  const int col = blockIdx.x * LT + l;
  const bool ok = col < m;
  const double* __restrict__ x0 = S[0].v[in_slot] + (ok ? col : m - 1);
  const T* __restrict__ pre = lane::twist<R>(g);
  rhs += col;
  if constexpr (B == 1) {
    T x[A];
    load_pairs<R, A>(x, x0, x0 + g.mn, m);
#pragma unroll
    for (int t = 0; t < n; ++t) x[t] = cmul(x[t], __ldg(&pre[t]));
    reg_dft<T, R, A>(x, false);
    if (ok) {
#pragma unroll
      for (int r = 0; r < n / 2; ++r) put_slot<R>(rhs, tab, kind, m, r, x[pos<A>(r)], x[pos<A>(n - 1 - r)]);
    }
  } else {
    T* ex = (T*)smem_raw + l;                        // position e of the line: ex[e LT]
#pragma unroll 1
    for (int t = grp; t < B; t += NG) {
      const double* __restrict__ p = x0 + (long long)t * m;
      T x[A];
      load_pairs<R, A>(x, p, p + g.mn, (long long)B * m);
#pragma unroll
      for (int q = 1; q < A; ++q) x[q] = cmul(x[q], root64<R>(q * (32 / A)));
      reg_dft<T, R, A>(x, false);
#pragma unroll
      for (int k = 0; k < A; ++k) ex[(t * A + k) * LT] = x[pos<A>(k)];
    }
    __syncthreads();
    // rows k1 and A-1-k1, whose twiddles are conjugate up to a shift by one slot (see k_lane_time)
#pragma unroll 1
    for (int k1 = grp; k1 < A / 2; k1 += NG) {
      T va[B], vb[B];
#pragma unroll
      for (int t = 0; t < B; ++t) {
        va[t] = ex[(t * A + k1) * LT];
        vb[t] = ex[(t * A + A - 1 - k1) * LT];
        if (t) {
          const T w = __ldg(&pre[t * (2 * k1 + 1)]);
          va[t] = cmul(va[t], w);
          vb[t] = lane::mulc(vb[t], w);
        }
      }
      reg_dft<T, R, B>(va, false);
      reg_dft<T, R, B>(vb, false);
      if (ok) {
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {             // slot k1 + A k2 or its partner, whichever is below n/2
          const T Xa = va[pos<B>(k2)], Xb = vb[pos<B>((B - k2) % B)];
          if (k2 < B / 2) put_slot<R>(rhs, tab, kind, m, k1 + A * k2, Xa, Xb);
          else put_slot<R>(rhs, tab, kind, m, n - 1 - k1 - A * k2, Xb, Xa);
        }
      }
    }
  }
}

// inverse: solutions of the n systems -> P^{-1} v (FP64, 2 halves)
template <typename R, int n>
__global__ void __launch_bounds__((mg_time_threads<R, n>()), (lane::time_blocks_per_sm<R, n, false>()))
    k_mg_time_inv(const Geom* __restrict__ G, const Slots* __restrict__ S, int out_slot, const cx<R>* __restrict__ tab,
                  int kind, const cx<R>* __restrict__ z) {
  using T = cx<R>;
  constexpr int A = lane::TimeShape<R, n>::A, B = lane::TimeShape<R, n>::B;
  constexpr int LT = mg_time_columns<R, n>(), NG = mg_time_threads<R, n>() / LT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geom& g = G[0];
  const int m = g.m, l = threadIdx.x % LT, grp = threadIdx.x / LT;
  const int col = blockIdx.x * LT + l;
  const bool ok = col < m;
  double* __restrict__ y = S[0].v[out_slot] + col;
  double* __restrict__ y2 = y + g.mn;
  const T* __restrict__ pre = lane::twist<R>(g);
  z += ok ? col : m - 1;
  const R sc = (R)1 / (R)n;
  unsigned rare = 0;
  if constexpr (B == 1) {
    T x[A];
#pragma unroll
    for (int r = 0; r < n / 2; ++r) get_slot<R>(z, tab, kind, m, r, x[r], x[n - 1 - r]);
    reg_dft<T, R, A>(x, true);
    if (!ok) return;
#pragma unroll
    for (int t = 0; t < n; ++t) {
      x[pos<A>(t)] = cscale(lane::mulc(x[pos<A>(t)], __ldg(&pre[t])), sc);
      store_pair<R>(y + (long long)t * m, y2 + (long long)t * m, x[pos<A>(t)], rare);
    }
    if (rare) {
#pragma unroll
      for (int t = 0; t < n; ++t) y2[(long long)t * m] = (double)x[pos<A>(t)].y;
    }
  } else {
    T* ex = (T*)smem_raw + l;
#pragma unroll 1
    for (int k1 = grp; k1 < A / 2; k1 += NG) {
      T za[B], zb[B];
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) {
        T Xr, Xq;
        if (k2 < B / 2) {
          get_slot<R>(z, tab, kind, m, k1 + A * k2, Xr, Xq);
          za[k2] = Xr;
          zb[(B - k2) % B] = Xq;
        } else {
          get_slot<R>(z, tab, kind, m, n - 1 - k1 - A * k2, Xr, Xq);
          za[k2] = Xq;
          zb[(B - k2) % B] = Xr;
        }
      }
      reg_dft<T, R, B>(za, true);
      reg_dft<T, R, B>(zb, true);
#pragma unroll
      for (int t = 0; t < B; ++t) {
        T a = za[pos<B>(t)], b = zb[pos<B>(t)];
        if (t) {
          const T w = __ldg(&pre[t * (2 * k1 + 1)]);
          a = lane::mulc(a, w);
          b = cmul(b, w);
        }
        ex[(t * A + k1) * LT] = cscale(a, sc);
        ex[(t * A + A - 1 - k1) * LT] = cscale(b, sc);
      }
    }
    __syncthreads();
    if (!ok) return;
#pragma unroll 1
    for (int t = grp; t < B; t += NG) {
      T x[A];
#pragma unroll
      for (int k = 0; k < A; ++k) x[k] = ex[(t * A + k) * LT];
      reg_dft<T, R, A>(x, true);
      rare = 0;
#pragma unroll
      for (int q = 0; q < A; ++q) {
        const long long at = (long long)(t + B * q) * m;
        if (q) x[pos<A>(q)] = lane::mulc(x[pos<A>(q)], root64<R>(q * (32 / A)));
        store_pair<R>(y + at, y2 + at, x[pos<A>(q)], rare);
      }
      if (rare) {
#pragma unroll
        for (int q = 0; q < A; ++q) y2[(long long)(t + B * q) * m] = (double)x[pos<A>(q)].y;
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// host orchestration
// ------------------------------------------------------------------------------------------
static unsigned blocks_for(long long len) { return (unsigned)((len + 255) / 256); }

// `base`: see k_mg_postsmooth (FP32 Dirichlet levels with a coarser one only)
template <typename R>
static void vcycle(const MgHost& h, const cx<R>* tab, int kind, int l, const cx<R>* rhs, cx<R>* z, cx<R>* spare,
                   cudaStream_t st, cx<R>* base = nullptr) {
  const MgLevel& L = h.lev[l];
  if (l > 0 && l == h.tail_l0) {      // the coarse levels in one launch, one block per slot
    MgTail T;
    for (int k = 0; k < h.nlev; ++k) T.lev[k] = h.lev[k];
    T.l0 = l; T.nlev = h.nlev;
    static DeviceOnce once;
    set_smem_limit(once, k_mg_vcycle_tail<R>, (int)kTailSmemMax);
    k_mg_vcycle_tail<R><<<h.nsys / 2, 256, tail_smem<R>(T), st>>>(T, tab, kind, rhs, z);
    g_mg_launches += 1;
    return;
  }
  const dim3 grids = grid_for(L.N, h.nsys / 2);     // one slot (two systems) per grid z
  const R w = (R)kJacobiWeight;
  if (l == h.nlev - 1) {
    if (L.neu) k_mg_coarse_neu<R><<<blocks_for((long long)h.nsys * 9), 256, 0, st>>>(L, h.nsys, tab, kind, rhs, z);
    else        // exact solve on the single-unknown grid: z = rhs / diag
      k_mg_jacobi<R, true><<<grids, kMgBlock, 0, st>>>(L, tab, kind, rhs, nullptr, z, (R)1);
    g_mg_launches += 1;
    return;
  }
  // FP32 on a Dirichlet level: one launch before the restriction and one after the coarse levels.  Not in
  // FP64: the fused kernels repeat the sweeps on their halos, and the FP64 rate bounds those (level 0 at
  // N = 255, n = 256: 2.32 ms fused against about 1.9 ms for the three launches of the pre-smoothing).
  if constexpr (sizeof(R) == 4 && kNu == 2) {
    if (!L.neu) {
      const MgLevel& C = h.lev[l + 1];
      const dim3 tiles = tile_grid(L.N, h.nsys / 2);
      k_mg_presmooth<R><<<tiles, kMgBlock, 0, st>>>(L, tab, kind, rhs, spare, z, w);    // solution, residual
      k_mg_restrict<R, false><<<grid_for(C.N, h.nsys / 2), kMgBlock, 0, st>>>(L.N, z, (cx<R>*)C.a[0]);
      vcycle<R>(h, tab, kind, l + 1, (cx<R>*)C.a[0], (cx<R>*)C.a[1], (cx<R>*)C.a[2], st);
      k_mg_postsmooth<R><<<tiles, kMgBlock, 0, st>>>(L, tab, kind, rhs, spare, (const cx<R>*)C.a[1], z, base, w);
      g_mg_launches += 3;
      return;
    }
  }
  // pre-smoothing from zero: the first sweep z1 = w D^{-1} rhs, then nu1 - 1 sweeps ping-ponging
  // between `spare` and z.  The nu1 + nu2 = 2 nu sweeps alternate between the two buffers, so
  // starting in `spare` leaves the last post-smoothing sweep in z.
  cx<R>* cur = spare;
  cx<R>* oth = z;
  k_mg_jacobi<R, true><<<grids, kMgBlock, 0, st>>>(L, tab, kind, rhs, nullptr, cur, w);
  for (int s = 1; s < kNu; ++s) {
    k_mg_jacobi<R, false><<<grids, kMgBlock, 0, st>>>(L, tab, kind, rhs, cur, oth, w);
    std::swap(cur, oth);
  }
  k_mg_resid<R><<<grids, kMgBlock, 0, st>>>(L, tab, kind, rhs, cur, oth);
  g_mg_launches += kNu + 1;
  // restrict the residual to the coarse right-hand side
  const MgLevel& C = h.lev[l + 1];
  const dim3 gridc = grid_for(C.N, h.nsys / 2);
  cx<R>* crhs = (cx<R>*)C.a[0];
  if (L.neu) k_mg_restrict<R, true><<<gridc, kMgBlock, 0, st>>>(L.N, oth, crhs);
  else k_mg_restrict<R, false><<<gridc, kMgBlock, 0, st>>>(L.N, oth, crhs);
  vcycle<R>(h, tab, kind, l + 1, crhs, (cx<R>*)C.a[1], (cx<R>*)C.a[2], st);
  if (L.neu) k_mg_prolong_add<R, true><<<grids, kMgBlock, 0, st>>>(L.N, (const cx<R>*)C.a[1], cur);
  else k_mg_prolong_add<R, false><<<grids, kMgBlock, 0, st>>>(L.N, (const cx<R>*)C.a[1], cur);
  for (int s = 0; s < kNu; ++s) {
    k_mg_jacobi<R, false><<<grids, kMgBlock, 0, st>>>(L, tab, kind, rhs, cur, oth, w);
    std::swap(cur, oth);
  }
  g_mg_launches += kNu + 2;
  if (cur != z) {
    const long long len = (long long)h.nsys * L.N * L.N;
    k_mg_axpy<R><<<blocks_for(len), 256, 0, st>>>(len, cur, z, 1);
    g_mg_launches += 1;
  }
}

template <typename R, int n>
static cudaError_t mg_apply(const Batch& B, const Geom& g, const MgHost& h, int kind, int cycles, int in_slot,
                            int out_slot) {
  using T = cx<R>;
  cudaStream_t st = B.stream;
  const T* tab = (const T*)(sizeof(R) == 4 ? (const void*)h.tab_f : (const void*)h.tab_d);
  const MgLevel& F = h.lev[0];
  const long long len = (long long)h.nsys * F.N * F.N;
  T* r0 = (T*)F.a[0];
  T* z0 = (T*)h.zfine;
  T* x0 = (T*)h.xfine;
  constexpr int cols = mg_time_columns<R, n>(), threads = mg_time_threads<R, n>();
  constexpr size_t smem = lane::time_smem<R, n, false>();
  static DeviceOnce once;
  once([] {
    cudaFuncSetAttribute(k_mg_time_fwd<R, n>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return cudaFuncSetAttribute(k_mg_time_inv<R, n>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  const unsigned tb = (unsigned)((g.m + cols - 1) / cols);
  k_mg_time_fwd<R, n><<<tb, threads, smem, st>>>(B.G, B.S, in_slot, tab, kind, r0);
  g_mg_launches += 2;
  for (int c = 0; c < cycles; ++c) {
    if (c == 0) {
      vcycle<R>(h, tab, kind, 0, r0, z0, (T*)F.a[1], st);
    } else {
      k_mg_resid<R><<<grid_for(F.N, h.nsys / 2), kMgBlock, 0, st>>>(F, tab, kind, r0, z0, x0);
      const bool adds = sizeof(R) == 4 && !F.neu && h.nlev > 1;   // the last kernel of the cycle adds to z0
      vcycle<R>(h, tab, kind, 0, x0, (T*)F.a[2], (T*)F.a[1], st, adds ? z0 : nullptr);
      if (!adds) k_mg_axpy<R><<<blocks_for(len), 256, 0, st>>>(len, (const T*)F.a[2], z0, 0);
      g_mg_launches += 1 + !adds;
    }
  }
  k_mg_time_inv<R, n><<<tb, threads, smem, st>>>(B.G, B.S, out_slot, tab, kind, z0);
  return cudaGetLastError();
}

template <typename R>
static cudaError_t mg_dispatch(const Batch& B, const Geom& g, const MgHost& h, int kind, int cycles, int in_slot,
                               int out_slot) {
  switch (g.n) {
    case 2: return mg_apply<R, 2>(B, g, h, kind, cycles, in_slot, out_slot);
    case 4: return mg_apply<R, 4>(B, g, h, kind, cycles, in_slot, out_slot);
    case 8: return mg_apply<R, 8>(B, g, h, kind, cycles, in_slot, out_slot);
    case 16: return mg_apply<R, 16>(B, g, h, kind, cycles, in_slot, out_slot);
    case 32: return mg_apply<R, 32>(B, g, h, kind, cycles, in_slot, out_slot);
    case 64: return mg_apply<R, 64>(B, g, h, kind, cycles, in_slot, out_slot);
    case 128: return mg_apply<R, 128>(B, g, h, kind, cycles, in_slot, out_slot);
    case 256: return mg_apply<R, 256>(B, g, h, kind, cycles, in_slot, out_slot);
    case 512: return mg_apply<R, 512>(B, g, h, kind, cycles, in_slot, out_slot);
    default: return cudaErrorInvalidValue;
  }
}

int mg_launch_count(int kind) { (void)kind; return 0; }
long long mg_launch_total() { return g_mg_launches; }

cudaError_t launch_precond_mg(const Batch& B, const Geom& g, int kind, int prec, int cycles, int in_slot,
                              int out_slot) {
  if (B.count != 1 || !g.mg) return cudaErrorInvalidValue;
  const MgHost* h = find_host(g.mg);
  if (!h) return cudaErrorInvalidValue;
  if (kind != PCB_PREC_PS && kind != PCB_PREC_PMS) return cudaErrorInvalidValue;
  return prec == PCB_MIXED ? mg_dispatch<float>(B, g, *h, kind, cycles, in_slot, out_slot)
                           : mg_dispatch<double>(B, g, *h, kind, cycles, in_slot, out_slot);
}

}  // namespace pcb
