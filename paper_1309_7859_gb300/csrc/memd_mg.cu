// memd_mg.cu -- the initial field and the effective permittivity through a
// scalar potential (Sec. II and Sec. V).
//
// The relaxed field is the minimiser of sum D^2 / 2 eps at fixed div D and
// fixed mean of D; at the minimum E = D / eps is curl free, i.e. a lattice
// gradient plus a constant: D = eps (-grad phi + E0).  phi solves the
// variable-coefficient Poisson problem L phi = -div(eps grad phi) = f on the
// periodic vertex lattice, and E0 follows from the mean of D through the
// effective permittivity, whose columns come from the three cell problems
// L psi_d = -div(eps e_d) (homogenisation).  The plaquette-rotation
// relaxation reaches the same minimiser; this is a faster route to it on
// V unknowns instead of 3V.
//
// Solver: conjugate gradients preconditioned by one symmetric multigrid
// V(2,2)-cycle, FP64 throughout, the whole solve in one cooperative launch.
// A level whose extents are all even coarsens geometrically (vertex-centred,
// by 2): red-black Gauss-Seidel, full-weighting restriction, trilinear
// prolongation, coarse link conductances from two fine links in series
// averaged over the 3 x 3 perpendicular neighbourhood.  A level with an odd
// extent coarsens by aggregating vertex pairs (a triple at the end of an odd
// axis): damped Jacobi, Galerkin coarse operator, piecewise-constant
// transfers with an over-corrected coarse correction.  The last level (an
// extent below 4, or at most 64 vertices) is swept.
//
// Every value and every sum is rounded in one fixed order, whatever the grid
// and the number of right-hand sides: B of a system one
// step from its relaxed field is nothing but the rounding of that field
// (curl E is zero in exact arithmetic), so a solver that is as accurate but
// rounds elsewhere gives every such B anew.  Sums therefore run in the order
// of the reductions of memd_setup.cu (304 blocks of 256 threads in turn over
// the vertices), and products that are fused with a sum are written so.
//
// What bounds it: the FP64 pipe of GB300 takes 16 cycles a warp instruction
// and a dependent one waits ~75, and below 10^5 vertices the latency of the
// phases: a grid barrier costs ~1.2 us where a kernel launch cost 2.5-4 us,
// and the host takes no part in the iteration.  Levels of at most
// kMgCtaSites vertices run in one CTA a right-hand side, which needs CTA
// barriers only; on levels with less work than the grid has warps each
// right-hand side gets warps of its own.  A whole system's setup (48^3, 2200
// charges; 77^3, 10^4 charges) takes 4.1 and 15.4 ms, with one launch a half
// sweep and host checks between iterations it took 8.6 and 27.0.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "memd_ctx.cuh"
#include "memd_internal.cuh"

namespace memd {

namespace {

// 512 threads with all the registers they take: held to 64 registers the
// three-right-hand-side solve spills, 1024 threads only add to the barriers
constexpr int kMgThreads = 512;
constexpr int kMgWarps = kMgThreads / 32;
constexpr int kMgMaxLevels = 32;  // an axis has less than 2^30 vertices
// Levels up to this size run in one CTA a right-hand side, in shared memory:
// a phase of 6^3 vertices takes ~0.9 us there and ~2.2 us with a grid barrier;
// from 8^3 on the one SM's FP64 pipe is the slower.  The last level is taken
// up to kMgCtaLast, its up to 48 half sweeps being barriers above all.
constexpr int kMgCtaSites = 256;
constexpr int kMgCtaLast = 1024;
constexpr int kMgCtaLevels = 8;
constexpr int kMgGrid = 256;  // most CTAs
// levels with so few vertices: each right-hand side by warps of its own
constexpr int kMgSplitSites = 50000;
constexpr int kMgQ = 9;       // most sums of one reduction
constexpr int kMgSlots = 7;   // one a use
constexpr unsigned long long kMgWaitNs = 2000000000ull;  // bound of a barrier wait
constexpr double kJacobi = 0.8;   // damping
constexpr double kAggAlpha = 1.6; // over-correction of the aggregated coarse correction

// the order of a sum over the vertices (memd_setup.cu's reductions): thread T
// of kSumThreads adds v = T, T + kSumThreads, ..., a warp its 32 by halves, a
// block its eight warps in turn, then 256 threads the blocks likewise
constexpr int kSumBlocks = 2 * 152;
constexpr int kSumWarps = 8 * kSumBlocks;
constexpr int kSumThreads = 32 * kSumWarps;

// n / d for 0 <= n < 2^31 (multiply and shift)
struct FastDiv {
  unsigned d, m, s;
};
FastDiv fast_div(unsigned d) {
  FastDiv f{d, 0, 0};
  while ((1ull << f.s) < d) ++f.s;
  f.m = (unsigned)(((1ull << 32) * ((1ull << f.s) - d)) / d + 1);
  return f;
}
__device__ __forceinline__ int operator/(int n, const FastDiv& f) {
  return (int)((__umulhi(f.m, (unsigned)n) + (unsigned)n) >> f.s);
}

// One level.  Right-hand side r of a multi-right-hand-side array is at r V.
struct MgLv {
  int n0, n1, n2, V;
  int rb;       // every extent even: red-black, geometric; else Jacobi, aggregation
  int split;    // each right-hand side by warps of its own
  FastDiv d0, d1, dh;  // by n0, n1, n0 / 2
  double* w;    // 3 V conductances of the links
  double* dg;   // V: their sum at a vertex
  double* idg;  // V: its inverse
  double* f;    // right-hand side
  double* r;    // residual
  double* phi;  // correction
  double* alt;  // Jacobi: every second sweep's
};

enum : int { kMgCells = 0, kMgRelax = 1 };

struct MgOut {
  double sum[9];    // cells: of flux component e of problem d at 3 e + d; relax: of the
                    // components of D64 at 0, of -eps grad phi at 3
  int converged, iters, timeout, pad;
};

struct MgArgs {
  int nl, nlg;  // levels, and how many of them are swept by the whole grid
  int maxit;
  double tol;
  double inv_a, inv_a2;
  const double* ie64;
  double* x;    // solution (cells: psi)
  double* p;
  double* q;    // shared with the residual of level 0, which the cycle leaves behind
  double* part;       // kMgSlots x kMgQ sums of every warp
  unsigned* arrivals; // barrier count, 0 at launch
  MgOut* out;
  double* D64;        // relax: in and out
  MgLv lv[kMgMaxLevels];
};

__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }

// n / d, correctly rounded, from y = 1 / d correctly rounded: with the
// quotient n y corrected once, the remainder of the second correction is exact
// and its quotient the rounded one (P. Markstein, IBM J. Res. Dev. 34, 1990).
// The bounds keep every term normal; outside them the division itself.
__device__ __noinline__ double quotient_slow(double n, double d) { return n / d; }
__device__ __forceinline__ bool mid_range(double x) {  // 2^-500 <= |x| < 2^500
  return (unsigned)((__double2hiint(x) & 0x7fffffff) - ((1023 - 500) << 20)) < 1000u << 20;
}
__device__ __forceinline__ double quotient(double n, double d, double y) {
  double q = mul_(n, y);
  if (!(mid_range(n) && mid_range(q)) && n != 0.0) return quotient_slow(n, d);
  q = fma_(fma_(-q, d, n), y, q);
  return fma_(fma_(-q, d, n), y, q);
}

struct Nb {
  int xp, xm, yp, ym, zp, zm;
};
__device__ __forceinline__ Nb neighbours(const MgLv& L, int v, int i, int j, int k) {
  const int P = L.n0 * L.n1;
  Nb b;
  b.xp = i + 1 == L.n0 ? v - i : v + 1;
  b.xm = i == 0 ? v + L.n0 - 1 : v - 1;
  b.yp = j + 1 == L.n1 ? v - j * L.n0 : v + L.n0;
  b.ym = j == 0 ? v + (L.n1 - 1) * L.n0 : v - L.n0;
  b.zp = k + 1 == L.n2 ? v - k * P : v + P;
  b.zm = k == 0 ? v + (L.n2 - 1) * P : v - P;
  return b;
}
__device__ __forceinline__ void coords(const MgLv& L, int v, int& i, int& j, int& k) {
  const int row = v / L.d0;
  i = v - row * L.n0;
  k = row / L.d1;
  j = row - k * L.n1;
}

// the links of a vertex, and the neighbours' weighted sum
struct Links {
  double xp, xm, yp, ym, zp, zm;
  __device__ __forceinline__ Links(const MgLv& L, int v, const Nb& b)
      : xp(L.w[v]), xm(L.w[b.xm]), yp(L.w[L.V + v]), ym(L.w[L.V + b.ym]), zp(L.w[2 * L.V + v]),
        zm(L.w[2 * L.V + b.zm]) {}
  __device__ __forceinline__ double sum() const {
    return add_(add_(add_(xp, xm), add_(yp, ym)), add_(zp, zm));
  }
  __device__ __forceinline__ double of(const double* p, const Nb& b) const {
    const double x = fma_(xp, p[b.xp], mul_(xm, p[b.xm]));
    const double y = fma_(yp, p[b.yp], mul_(ym, p[b.ym]));
    const double z = fma_(zp, p[b.zp], mul_(zm, p[b.zm]));
    return add_(add_(x, y), z);
  }
};

// ---------------------------------------------------------- phases
// t0, stride: this thread's share of the vertices; r0: first right-hand side

// Gauss-Seidel on the vertices of one colour ((i + j + k) mod 2)
template <int NR>
__device__ __forceinline__ void sweep(const MgLv& L, int c, int t0, int stride, int r0) {
  const int hx = L.n0 / 2, H = L.V / 2, V = L.V;
  for (int h = t0; h < H; h += stride) {
    const int row = h / L.dh;
    const int k = row / L.d1, j = row - k * L.n1;
    const int i = 2 * (h - row * hx) + ((c + j + k) & 1);
    const int v = i + L.n0 * row;
    const Nb b = neighbours(L, v, i, j, k);
    const Links w(L, v, b);
    const double dg = L.dg[v], id = L.idg[v];
    double y[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r)
      y[r] = quotient(add_(L.f[(r0 + r) * V + v], w.of(L.phi + (r0 + r) * V, b)), dg, id);
#pragma unroll
    for (int r = 0; r < NR; ++r) L.phi[(r0 + r) * V + v] = y[r];
  }
}

// damped Jacobi: to = from + omega (f - L from) / diag
template <int NR>
__device__ __forceinline__ void jacobi(const MgLv& L, const double* from, double* to, int t0,
                                       int stride, int r0) {
  const int V = L.V;
  for (int v = t0; v < V; v += stride) {
    int i, j, k;
    coords(L, v, i, j, k);
    const Nb b = neighbours(L, v, i, j, k);
    const Links w(L, v, b);
    const double dg = L.dg[v], id = L.idg[v];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const double* p = from + (r0 + r) * V;
      const double a = fma_(dg, p[v], -w.of(p, b));
      to[(r0 + r) * V + v] =
          fma_(kJacobi, quotient(sub_(L.f[(r0 + r) * V + v], a), dg, id), p[v]);
    }
  }
}

// the first sweep from zero at one vertex: the first colour's values (the
// second's are overwritten unread), or the whole Jacobi sweep
__device__ __forceinline__ void first_sweep(const MgLv& L, int at, int v, int i, int j, int k,
                                            double f) {
  if (L.rb) {
    if (((i + j + k) & 1) == 0) L.phi[at] = quotient(add_(f, 0.0), L.dg[v], L.idg[v]);
  } else {
    L.alt[at] = mul_(kJacobi, quotient(f, L.dg[v], L.idg[v]));
  }
}

// f - L phi
template <int NR>
__device__ __forceinline__ void residual(const MgLv& L, int t0, int stride, int r0) {
  const int V = L.V;
  for (int v = t0; v < V; v += stride) {
    int i, j, k;
    coords(L, v, i, j, k);
    const Nb b = neighbours(L, v, i, j, k);
    const Links w(L, v, b);
    const double dg = L.dg[v];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const double* p = L.phi + (r0 + r) * V;
      L.r[(r0 + r) * V + v] = sub_(L.f[(r0 + r) * V + v], fma_(dg, p[v], -w.of(p, b)));
    }
  }
}

// Aggregates: coarse vertex I along an axis of n fine vertices and m = n / 2
// coarse ones holds fine 2I, 2I + 1, and also 2I + 2 when it is the last one
// of an odd n.
__device__ __forceinline__ int agg_hi(int I, int m, int n) { return I == m - 1 ? n - 1 : 2 * I + 1; }
__device__ __forceinline__ int agg_of(int i, int m) { return min(i >> 1, m - 1); }

// f of the coarse level and its first sweep from zero.  Geometric: sum_o
// prod_d (1 - |o_d| / 2) / 8 r(2 I + o); aggregation: the sum of the aggregate.
template <int NR>
__device__ __forceinline__ void restrict_to(const MgLv& F, const MgLv& C, bool first, int t0,
                                            int stride, int r0) {
  for (int v = t0; v < C.V; v += stride) {
    int I, J, K;
    coords(C, v, I, J, K);
    double s[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) s[r] = 0.0;
    if (F.rb) {
      const int x[3] = {I == 0 ? F.n0 - 1 : 2 * I - 1, 2 * I, 2 * I + 1};
      const int y[3] = {J == 0 ? F.n1 - 1 : 2 * J - 1, 2 * J, 2 * J + 1};
      const int z[3] = {K == 0 ? F.n2 - 1 : 2 * K - 1, 2 * K, 2 * K + 1};
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const int row = F.n0 * (y[b] + F.n1 * z[c]);
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const double wt = (a == 1 ? 1.0 : 0.5) * (b == 1 ? 1.0 : 0.5) * (c == 1 ? 1.0 : 0.5);
#pragma unroll
            for (int r = 0; r < NR; ++r) s[r] = fma_(wt, F.r[(r0 + r) * F.V + row + x[a]], s[r]);
          }
        }
#pragma unroll
      for (int r = 0; r < NR; ++r) s[r] = mul_(0.125, s[r]);
    } else {
      const int i1 = agg_hi(I, C.n0, F.n0), j1 = agg_hi(J, C.n1, F.n1), k1 = agg_hi(K, C.n2, F.n2);
      for (int k = 2 * K; k <= k1; ++k)
        for (int j = 2 * J; j <= j1; ++j)
          for (int i = 2 * I; i <= i1; ++i)
#pragma unroll
            for (int r = 0; r < NR; ++r)
              s[r] = add_(s[r], F.r[(r0 + r) * F.V + i + F.n0 * (j + F.n1 * k)]);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      C.f[(r0 + r) * C.V + v] = s[r];
      if (first) first_sweep(C, (r0 + r) * C.V + v, v, I, J, K, s[r]);
    }
  }
}

// phi += coarse correction.  Geometric: trilinear, and only on the first
// colour (the half sweep that follows overwrites the second): a thread takes
// the four such vertices 2 I + {0, 1}^3 of a coarse one.
template <int NR>
__device__ __forceinline__ void prolong(const MgLv& F, const MgLv& C, int t0, int stride, int r0) {
  if (!F.rb) {
    for (int v = t0; v < F.V; v += stride) {
      int i, j, k;
      coords(F, v, i, j, k);
      const int u = agg_of(i, C.n0) + C.n0 * (agg_of(j, C.n1) + C.n1 * agg_of(k, C.n2));
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        double* p = F.phi + (r0 + r) * F.V + v;
        *p = fma_(kAggAlpha, C.phi[(r0 + r) * C.V + u], *p);
      }
    }
    return;
  }
  for (int v = t0; v < C.V; v += stride) {
    int I, J, K;
    coords(C, v, I, J, K);
    const int I1 = I + 1 == C.n0 ? 0 : I + 1, J1 = J + 1 == C.n1 ? 0 : J + 1,
              K1 = K + 1 == C.n2 ? 0 : K + 1;
    const int c00 = C.n0 * (J + C.n1 * K), c10 = C.n0 * (J1 + C.n1 * K),
              c01 = C.n0 * (J + C.n1 * K1), c11 = C.n0 * (J1 + C.n1 * K1);
    const int u = 2 * I + F.n0 * (2 * J + F.n1 * 2 * K);
    const int sy = F.n0, sz = F.n0 * F.n1;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const double* e = C.phi + (r0 + r) * C.V;
      double* p = F.phi + (r0 + r) * F.V + u;
      const double a0 = p[0], a1 = p[1 + sy], a2 = p[1 + sz], a3 = p[sy + sz];
      const double e0 = e[c00 + I], x = add_(e0, e[c00 + I1]), ey = e[c10 + I], ez = e[c01 + I];
      p[0] = add_(a0, e0);
      p[1 + sy] = fma_(0.25, add_(add_(x, ey), e[c10 + I1]), a1);
      p[1 + sz] = fma_(0.25, add_(add_(x, ez), e[c01 + I1]), a2);
      p[sy + sz] = fma_(0.25, add_(add_(add_(e0, ey), ez), e[c11 + I]), a3);
    }
  }
}

// Conductance of link d of coarse vertex (I, J, K).  Geometric: the two fine
// d-links from 2I + o (o perpendicular to d) in series, averaged with weights
// (1/4, 1/2, 1/4)^2 over o, halved for the coarse spacing; aggregation: the
// sum of the fine d-links that leave the aggregate towards the next.
__device__ __forceinline__ double coarse_link(const MgLv& F, const MgLv& C, int d, int I, int J,
                                              int K) {
  const int c[3] = {I, J, K}, nf[3] = {F.n0, F.n1, F.n2}, nc[3] = {C.n0, C.n1, C.n2};
  const double* w = F.w + (int64_t)d * F.V;
  double s = 0.0;
  if (F.rb) {
    const int e1 = (d + 1) % 3, e2 = (d + 2) % 3;
    const int st[3] = {1, F.n0, F.n0 * F.n1};
    const int base = 2 * c[d] * st[d];
    for (int b = -1; b <= 1; ++b)
      for (int a = -1; a <= 1; ++a) {
        const int p1 = 2 * c[e1] + a, p2 = 2 * c[e2] + b;
        const int v = base + (p1 < 0 ? p1 + nf[e1] : p1) * st[e1] + (p2 < 0 ? p2 + nf[e2] : p2) * st[e2];
        const double w1 = w[v], w2 = w[v + st[d]];
        const double ser = mul_(w1, w2) / add_(w1, w2);
        s = fma_((a ? 0.5 : 1.0) * (b ? 0.5 : 1.0) * 0.25, ser, s);
      }
    return mul_(0.5, s);
  }
  int lo[3], hi[3];
  for (int e = 0; e < 3; ++e) {
    lo[e] = 2 * c[e];
    hi[e] = agg_hi(c[e], nc[e], nf[e]);
  }
  lo[d] = hi[d];
  for (int k = lo[2]; k <= hi[2]; ++k)
    for (int j = lo[1]; j <= hi[1]; ++j)
      for (int i = lo[0]; i <= hi[0]; ++i) s = add_(s, w[i + F.n0 * (j + F.n1 * k)]);
  return s;
}

// ------------------------------------------------------- barrier and sums
// Grid barrier of the cooperative launch over a count of arrivals that only
// grows (0 at launch): complete when it reaches round x CTAs.  The wait is
// bounded; a CTA that gives up marks the result and every CTA leaves.
struct GridSync {
  unsigned* arrivals;
  MgOut* out;
  unsigned target;
  int* s_ok;
  __device__ bool operator()() {
    __syncthreads();
    if (gridDim.x == 1) return true;
    target += gridDim.x;
    if (threadIdx.x == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrivals) : "memory");
      int ok = 1;
      unsigned long long t0 = 0, t;
      for (unsigned it = 1;; ++it) {
        unsigned cur;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(arrivals) : "memory");
        if (cur >= target) break;
        if ((it & 255u) == 0u) {
          asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
          if (t0 == 0) t0 = t;
          if (t - t0 > kMgWaitNs || __ldcg(&out->timeout) != 0) {
            atomicExch(&out->timeout, 1);
            ok = 0;
            break;
          }
        }
      }
      *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
  }
};

// NQ sums of warp W of the order above into slot (every lane calls it); every
// CTA forms the totals after the next grid barrier.  nW: the warps that have
// a vertex.
template <int NQ>
__device__ __forceinline__ void share_sums(double* part, int slot, int W, int nW,
                                           const double (&x)[NQ]) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    double s = x[q];
    for (int o = 16; o > 0; o >>= 1) s = add_(s, __shfl_down_sync(0xffffffffu, s, o));
    if ((threadIdx.x & 31) == 0) part[(slot * kMgQ + q) * nW + W] = s;
  }
}
struct SumScratch {
  double blk[kMgQ][kSumBlocks];
  double warp[kMgQ][8];
  double tot[kMgQ];
};
template <int NQ>
__device__ __forceinline__ void total_sums(const double* part, int slot, int nW, double (&x)[NQ],
                                           SumScratch& sh) {
  for (int t = threadIdx.x; t < NQ * kSumBlocks; t += kMgThreads) {
    const int q = t / kSumBlocks, b = t - q * kSumBlocks;
    const double* p = part + (slot * kMgQ + q) * nW + 8 * b;
    double y[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) y[j] = 8 * b + j < nW ? __ldcg(p + j) : 0.0;
    double s = y[0];
    if (8 * b + 1 < nW)
#pragma unroll
      for (int j = 1; j < 8; ++j) s = add_(s, y[j]);
    sh.blk[q][b] = s;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 7, t = threadIdx.x & 255;
  for (int q = threadIdx.x >> 8; q < NQ; q += kMgThreads / 256) {
    double s = sh.blk[q][t];
    if (t + 256 < kSumBlocks) s = add_(s, sh.blk[q][t + 256]);
    for (int o = 16; o > 0; o >>= 1) s = add_(s, __shfl_down_sync(0xffffffffu, s, o));
    if (lane == 0) sh.warp[q][w] = s;
  }
  __syncthreads();
  if (threadIdx.x < NQ) {
    double s = sh.warp[threadIdx.x][0];
    for (int j = 1; j < 8; ++j) s = add_(s, sh.warp[threadIdx.x][j]);
    sh.tot[threadIdx.x] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) x[q] = sh.tot[q];
}

// sweeps each way on the last level
__device__ __forceinline__ int last_sweeps(const MgLv& L) { return L.V <= 512 ? 8 : 12; }
// half sweep s of the last level's forward and backward red-black sweeps
__device__ __forceinline__ int last_colour(int s, int sweeps) {
  return s < 2 * sweeps ? s & 1 : 1 - (s & 1);
}

// One V-cycle of right-hand side r on the levels of the one-CTA part (in
// shared memory, lv[0] .. lv[nc - 1]); top: the first of them in memory.
__device__ __forceinline__ void cta_cycle(const MgLv* lv, int nc, const MgLv& top, int r) {
  const int t = threadIdx.x;
  for (int v = t; v < top.V; v += kMgThreads) {
    int i, j, k;
    coords(top, v, i, j, k);
    const double f = top.f[r * top.V + v];
    lv[0].f[v] = f;
    first_sweep(lv[0], v, v, i, j, k, f);
  }
  __syncthreads();
  for (int l = 0; l + 1 < nc; ++l) {
    const MgLv& F = lv[l];
    if (F.rb) {
      for (int s = 1; s < 4; ++s) {
        sweep<1>(F, s & 1, t, kMgThreads, 0);
        __syncthreads();
      }
    } else {
      jacobi<1>(F, F.alt, F.phi, t, kMgThreads, 0);
      __syncthreads();
    }
    residual<1>(F, t, kMgThreads, 0);
    __syncthreads();
    restrict_to<1>(F, lv[l + 1], true, t, kMgThreads, 0);
    __syncthreads();
  }
  {
    const MgLv& L = lv[nc - 1];
    const int n = last_sweeps(L);
    if (L.rb) {
      for (int s = 1; s < 4 * n; ++s) {
        sweep<1>(L, last_colour(s, n), t, kMgThreads, 0);
        __syncthreads();
      }
    } else {
      for (int s = 1; s < 2 * n; ++s) {
        jacobi<1>(L, s & 1 ? L.alt : L.phi, s & 1 ? L.phi : L.alt, t, kMgThreads, 0);
        __syncthreads();
      }
    }
  }
  for (int l = nc - 2; l >= 0; --l) {
    const MgLv& F = lv[l];
    prolong<1>(F, lv[l + 1], t, kMgThreads, 0);
    __syncthreads();
    if (F.rb) {
      for (int s = 1; s < 5; ++s) {
        sweep<1>(F, s & 1, t, kMgThreads, 0);
        __syncthreads();
      }
    } else {
      jacobi<1>(F, F.phi, F.alt, t, kMgThreads, 0);
      __syncthreads();
      jacobi<1>(F, F.alt, F.phi, t, kMgThreads, 0);
      __syncthreads();
    }
  }
  for (int v = t; v < top.V; v += kMgThreads) top.phi[r * top.V + v] = lv[0].phi[v];
}

// The whole solve for NR right-hand sides.
//   cells: L psi_d = -div(eps e_d) for d < NR, psi_d of zero mean and the
//   sums of the fluxes eps_e (delta_ed - grad_e psi_d)
//   relax: L phi = div D64; D64 <- -eps grad phi, and the sums of D64 before
//   and after
// The residual is looked at every second iteration.  Stops when |r| <= tol
// |f| (2-norms) or, once the recursion has reached its rounding floor and
// |r|^2 grows again (to 100 times its least value), when that least value was
// below 1e4 tol^2 |f|^2.
template <int NR, int MODE>
__global__ void __launch_bounds__(kMgThreads, 1) k_mg_solve(const __grid_constant__ MgArgs a) {
  extern __shared__ double s_mem[];  // the levels of the one-CTA part
  __shared__ SumScratch sums;
  __shared__ MgLv s_lv[kMgCtaLevels];
  __shared__ int s_ok;
  GridSync grid{a.arrivals, a.out, 0u, &s_ok};
#define MG_GRID() \
  if (!grid()) return
  // neighbouring warps of work go to different SMs: a level with less work
  // than the grid has warps still uses every FP64 pipe
  const int lane = threadIdx.x & 31;
  const int w0 = (threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x;
  const int nwarps = (int)gridDim.x * kMgWarps;
  const int t0 = w0 * 32 + lane, stride = nwarps * 32;
  // a right-hand side's own warps (the level's split)
  const int own = nwarps / NR, sr = w0 / own, s0 = (w0 - sr * own) * 32 + lane, sstride = own * 32;
#define MG_EACH(L, fn, ...)                                    \
  do {                                                         \
    if (NR > 1 && (L).split) {                                 \
      if (sr < NR) fn<1>(__VA_ARGS__, s0, sstride, sr);        \
    } else {                                                   \
      fn<NR>(__VA_ARGS__, t0, stride, 0);                      \
    }                                                          \
  } while (0)
  const MgLv& L = a.lv[0];
  const int V = L.V, nW = min(kSumWarps, (V + 31) / 32);
  const double inv_a = a.inv_a, nV = (double)V;
  // vertices of warp W in the order of the sums
#define MG_WARPS(W) for (int W = w0; W < nW; W += nwarps)
#define MG_VERTICES(v, W) for (int v = 32 * W + lane; v < V; v += kSumThreads)
  double before[3] = {0.0, 0.0, 0.0};  // relax: sums of D64
  {
    // conductances of the finest level, the right-hand side and its sum
    constexpr int NQ = MODE == kMgRelax ? 4 : NR, kD = NQ == 4 ? 1 : 0;
    MG_WARPS(W) {
      double s[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) s[q] = 0.0;
      MG_VERTICES(v, W) {
        int i, j, k;
        coords(L, v, i, j, k);
        const Nb b = neighbours(L, v, i, j, k);
        const int vm[3] = {b.xm, b.ym, b.zm};
#pragma unroll
        for (int d = 0; d < 3; ++d) L.w[d * V + v] = a.inv_a2 / a.ie64[(int64_t)d * V + v];
        if (MODE == kMgRelax) {
          double dd[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const double D = a.D64[(int64_t)d * V + v];
            s[kD + d] = add_(s[kD + d], D);
            dd[d] = sub_(D, a.D64[(int64_t)d * V + vm[d]]);
          }
          const double f = mul_(inv_a, add_(add_(dd[0], dd[1]), dd[2]));
          L.f[v] = f;
          s[0] = add_(s[0], f);
        } else {
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            const double* ie = a.ie64 + (int64_t)r * V;
            const double f = mul_(-sub_(__drcp_rn(ie[v]), __drcp_rn(ie[vm[r]])), inv_a);
            L.f[r * V + v] = f;
            s[r] = add_(s[r], f);
          }
        }
      }
      share_sums<NQ>(a.part, 0, W, nW, s);
    }
    MG_GRID();
    double m[NQ];
    total_sums<NQ>(a.part, 0, nW, m, sums);
    if (MODE == kMgRelax) {
#pragma unroll
      for (int d = 0; d < 3; ++d) before[d] = m[kD + d];
    }
    // of zero mean, and its square
    MG_WARPS(W) {
      double s[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) s[r] = 0.0;
      MG_VERTICES(v, W)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double f = sub_(L.f[r * V + v], m[r] / nV);
        L.f[r * V + v] = f;
        s[r] = fma_(f, f, s[r]);
      }
      share_sums<NR>(a.part, 1, W, nW, s);
    }
  }
  // diagonals, and the conductances level by level
  for (int l = 0; l < a.nl; ++l) {
    const MgLv& F = a.lv[l];
    for (int v = t0; v < F.V; v += stride) {
      int i, j, k;
      coords(F, v, i, j, k);
      const double dg = Links(F, v, neighbours(F, v, i, j, k)).sum();
      F.dg[v] = dg;
      F.idg[v] = 1.0 / dg;
    }
    if (l + 1 < a.nl) {
      const MgLv& C = a.lv[l + 1];
      for (int t = t0; t < 3 * C.V; t += stride) {
        const int d = t >= 2 * C.V ? 2 : (t >= C.V ? 1 : 0);
        int I, J, K;
        coords(C, t - d * C.V, I, J, K);
        C.w[t] = coarse_link(F, C, d, I, J, K);
      }
    }
    MG_GRID();
  }
  double f2[NR], least[NR], rz[NR];
  bool done[NR];
  total_sums<NR>(a.part, 1, nW, f2, sums);
  bool all = true;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    done[r] = f2[r] == 0.0;
    least[r] = f2[r];
    rz[r] = 0.0;
    all = all && done[r];
  }
  // x = 0, the first sweep of level 0
  const bool grid0 = a.nlg > 0;
  for (int v = t0; v < V; v += stride) {
    int i, j, k;
    coords(L, v, i, j, k);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      a.x[r * V + v] = 0.0;
      if (grid0) first_sweep(L, r * V + v, v, i, j, k, L.f[r * V + v]);
    }
  }
  // the levels of the one-CTA part: coefficients into shared memory
  const int nc = a.nl - a.nlg;
  if (nc > 0 && (int)blockIdx.x < NR) {
    int at = 0;
    for (int l = 0; l < nc; ++l) {
      const MgLv& F = a.lv[a.nlg + l];
      const int U = F.V;
      double* b = s_mem + 9 * at;
      at += U;
      for (int v = threadIdx.x; v < U; v += kMgThreads) {
#pragma unroll
        for (int d = 0; d < 3; ++d) b[d * U + v] = F.w[d * U + v];
        b[3 * U + v] = F.dg[v];
        b[4 * U + v] = F.idg[v];
      }
      if (threadIdx.x == 0) {
        MgLv C = F;
        C.w = b;
        C.dg = b + 3 * U;
        C.idg = b + 4 * U;
        C.f = b + 5 * U;
        C.r = b + 6 * U;
        C.phi = b + 7 * U;
        C.alt = b + 8 * U;
        s_lv[l] = C;
      }
    }
    __syncthreads();
  }
  MG_GRID();
  int its = 0;
  const double tol2 = mul_(a.tol, a.tol);
  while (!all && its < a.maxit) {
    // z = M r in phi of level 0: one V-cycle, its first sweep made where r was
    for (int l = 0; l < a.nlg; ++l) {
      const MgLv& F = a.lv[l];
      if (l + 1 == a.nl) {  // the last level, too large for one CTA
        const int n = last_sweeps(F);
        for (int s = 1; s < (F.rb ? 4 : 2) * n; ++s) {
          if (F.rb)
            MG_EACH(F, sweep, F, last_colour(s, n));
          else
            MG_EACH(F, jacobi, F, s & 1 ? F.alt : F.phi, s & 1 ? F.phi : F.alt);
          MG_GRID();
        }
        break;
      }
      if (F.rb) {
        for (int s = 1; s < 4; ++s) {
          MG_EACH(F, sweep, F, s & 1);
          MG_GRID();
        }
      } else {
        MG_EACH(F, jacobi, F, F.alt, F.phi);
        MG_GRID();
      }
      MG_EACH(F, residual, F);
      MG_GRID();
      MG_EACH(F, restrict_to, F, a.lv[l + 1], l + 1 < a.nlg);
      MG_GRID();
    }
    if (nc > 0) {
      if ((int)blockIdx.x < NR) cta_cycle(s_lv, nc, a.lv[a.nlg], blockIdx.x);
      MG_GRID();
    }
    for (int l = (nc > 0 ? a.nlg : a.nl - 1) - 1; l >= 0; --l) {
      const MgLv& F = a.lv[l];
      MG_EACH(F, prolong, F, a.lv[l + 1]);
      MG_GRID();
      if (F.rb) {
        for (int s = 1; s < 5; ++s) {
          MG_EACH(F, sweep, F, s & 1);
          MG_GRID();
        }
      } else {
        MG_EACH(F, jacobi, F, F.phi, F.alt);
        MG_GRID();
        MG_EACH(F, jacobi, F, F.alt, F.phi);
        MG_GRID();
      }
    }
    // r . z
    MG_WARPS(W) {
      double s[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) s[r] = 0.0;
      MG_VERTICES(v, W)
#pragma unroll
      for (int r = 0; r < NR; ++r) s[r] = fma_(L.f[r * V + v], L.phi[r * V + v], s[r]);
      share_sums<NR>(a.part, 2, W, nW, s);
    }
    MG_GRID();
    double rz1[NR];
    total_sums<NR>(a.part, 2, nW, rz1, sums);
    // p = z + beta p (z at first), then q = L p and p . q
    double beta[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      beta[r] = rz[r] != 0.0 ? rz1[r] / rz[r] : 0.0;
      rz[r] = rz1[r];
    }
    // (a few vertices a thread at once: every load before the first store)
    constexpr int UP = NR == 1 ? 4 : 2;
    for (int v0 = t0; v0 < V; v0 += UP * stride) {
      double p[UP][NR], z[UP][NR];
#pragma unroll
      for (int u = 0; u < UP; ++u)
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int v = v0 + u * stride;
          const bool in = v < V;
          p[u][r] = in && its > 0 ? a.p[r * V + v] : 0.0;
          z[u][r] = in ? L.phi[r * V + v] : 0.0;
        }
#pragma unroll
      for (int u = 0; u < UP; ++u)
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (v0 + u * stride < V)
            a.p[r * V + v0 + u * stride] = its > 0 ? fma_(beta[r], p[u][r], z[u][r]) : z[u][r];
    }
    MG_GRID();
    MG_WARPS(W) {
      double pq[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) pq[r] = 0.0;
      MG_VERTICES(v, W) {
        int i, j, k;
        coords(L, v, i, j, k);
        const Nb b = neighbours(L, v, i, j, k);
        const Links w(L, v, b);
        const double dg = L.dg[v];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const double* p = a.p + r * V;
          const double s = fma_(dg, p[v], -w.of(p, b));
          a.q[r * V + v] = s;
          pq[r] = fma_(p[v], s, pq[r]);
        }
      }
      share_sums<NR>(a.part, 3, W, nW, pq);
    }
    MG_GRID();
    double alpha[NR];
    total_sums<NR>(a.part, 3, nW, alpha, sums);
    // x and r (of a problem that has arrived, as they are), and the next
    // cycle's first sweep
#pragma unroll
    for (int r = 0; r < NR; ++r)
      alpha[r] = !done[r] && alpha[r] != 0.0 ? rz[r] / alpha[r] : 0.0;
    constexpr int UX = NR == 1 ? 3 : 1;
    MG_WARPS(W) {
      double rr[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) rr[r] = 0.0;
      for (int v0 = 32 * W + lane; v0 < V; v0 += UX * kSumThreads) {
        double x[UX][NR], p[UX][NR], f[UX][NR], q[UX][NR];
#pragma unroll
        for (int u = 0; u < UX; ++u) {
          const int v = v0 + u * kSumThreads;
          const bool in = v < V;
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            x[u][r] = in ? a.x[r * V + v] : 0.0;
            p[u][r] = in ? a.p[r * V + v] : 0.0;
            f[u][r] = in ? L.f[r * V + v] : 0.0;
            q[u][r] = in ? a.q[r * V + v] : 0.0;
          }
        }
#pragma unroll
        for (int u = 0; u < UX; ++u) {
          const int v = v0 + u * kSumThreads;
          if (v >= V) break;
          int i, j, k;
          coords(L, v, i, j, k);
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            const double t = fma_(-alpha[r], q[u][r], f[u][r]);
            rr[r] = fma_(t, t, rr[r]);
            a.x[r * V + v] = fma_(alpha[r], p[u][r], x[u][r]);
            L.f[r * V + v] = t;
            if (grid0) first_sweep(L, r * V + v, v, i, j, k, t);
          }
        }
      }
      share_sums<NR>(a.part, 4, W, nW, rr);
    }
    MG_GRID();
    if (++its & 1) continue;
    double rr[NR];
    total_sums<NR>(a.part, 4, nW, rr, sums);
    all = true;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (!done[r]) {
        done[r] = rr[r] <= mul_(tol2, f2[r]) ||
                  (rr[r] > mul_(100.0, least[r]) &&
                   least[r] <= mul_(mul_(mul_(1e4, a.tol), a.tol), f2[r]));
        least[r] = rr[r] < least[r] ? rr[r] : least[r];
      }
      all = all && done[r];
    }
  }
  // x of zero mean
  double m[NR];
  MG_WARPS(W) {
    double s[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) s[r] = 0.0;
    MG_VERTICES(v, W)
#pragma unroll
    for (int r = 0; r < NR; ++r) s[r] = add_(s[r], a.x[r * V + v]);
    share_sums<NR>(a.part, 5, W, nW, s);
  }
  MG_GRID();
  total_sums<NR>(a.part, 5, nW, m, sums);
  for (int v = t0; v < V; v += stride)
#pragma unroll
    for (int r = 0; r < NR; ++r) a.x[r * V + v] = sub_(a.x[r * V + v], m[r] / nV);
  MG_GRID();
  // the fluxes eps (e_d - grad x), in the relaxation -eps grad x in D64 (left
  // as it came when the solve has not converged)
  if (MODE == kMgRelax && !all) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.out->iters = its;
    return;
  }
  double s[3 * NR];
  MG_WARPS(W) {
#pragma unroll
    for (int q = 0; q < 3 * NR; ++q) s[q] = 0.0;
    MG_VERTICES(v, W) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const int vp[3] = {b.xp, b.yp, b.zp};
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const double ie = a.ie64[(int64_t)e * V + v];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const double* p = a.x + r * V;
          const double g = MODE == kMgCells && e == r ? 1.0 : 0.0;
          const double F = fma_(-sub_(p[vp[e]], p[v]), inv_a, g) / ie;
          if (MODE == kMgRelax) a.D64[(int64_t)e * V + v] = F;
          s[3 * r + e] = add_(s[3 * r + e], F);
        }
      }
    }
    share_sums<3 * NR>(a.part, 6, W, nW, s);
  }
  MG_GRID();
  total_sums<3 * NR>(a.part, 6, nW, s, sums);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      if (MODE == kMgRelax) {
        a.out->sum[e] = before[e];
        a.out->sum[3 + e] = s[e];
      } else {
#pragma unroll
        for (int r = 0; r < NR; ++r) a.out->sum[3 * e + r] = s[3 * r + e];
      }
    }
    a.out->converged = all ? 1 : 0;
    a.out->iters = its;
  }
#undef MG_GRID
#undef MG_EACH
#undef MG_WARPS
#undef MG_VERTICES
}

// D64 += sum_d E0_d eps (e_d - grad psi_d)
struct MgE0 {
  double e[3];
};
__global__ void k_mg_mean_field(const __grid_constant__ MgLv L, const double* __restrict__ ie64,
                                const double* __restrict__ psi, MgE0 E0, double inv_a,
                                double* __restrict__ D64) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x, V = L.V;
  if (v >= V) return;
  int i, j, k;
  coords(L, v, i, j, k);
  const Nb b = neighbours(L, v, i, j, k);
  const int vp[3] = {b.xp, b.yp, b.zp};
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const int64_t t = (int64_t)e * V + v;
    const double ie = ie64[t];
    double D = D64[t];
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (E0.e[d] != 0.0) {
        const double* p = psi + (int64_t)d * V;
        D = fma_(E0.e[d], fma_(-sub_(p[vp[e]], p[v]), inv_a, e == d ? 1.0 : 0.0) / ie, D);
      }
    D64[t] = D;
  }
}

// ---------------------------------------------------------------- host
// A cooperative grid starts when all of it fits, whatever else is resident or
// queued on other streams (checked on GB300: two grids that each need every
// SM, the second at a higher priority, while a third kernel holds half of
// them: neither started in part), so concurrent solves and single-launch
// steps never hold SMs that another's barriers wait for.  Were one ever to
// start in part, its bounded waits end it, and the caller relaxes the field
// instead.
template <int NR, int MODE>
cudaError_t launch_solve(const MgArgs& a, int grid, size_t smem, cudaStream_t st) {
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_mg_solve<NR, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(9 * kMgCtaLast * sizeof(double)));
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kMgThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mg_solve<NR, MODE>, a);
}

// The levels and their scratch for NR right-hand sides, one block of memory.
struct MgPlan {
  MgArgs a{};
  double* block = nullptr;
  size_t zero_bytes = 0;  // the leading words cleared before a launch
  size_t smem = 0;
  int grid = 0;

  // x: the cell problems' potentials, or null for one of the plan's own
  bool build(memd_ctx* c, int nr, double* x) {
    const Mesh& m = c->mesh;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess)
      return false;
    // a warp of work for every warp of the grid on the finest level, one CTA an SM at most
    grid = (int)std::min<int64_t>(std::min(sms, kMgGrid), std::max<int64_t>(nr, (m.V + 127) / 128));
    int n[3] = {m.n[0], m.n[1], m.n[2]};
    size_t words = 0;
    std::vector<size_t> at;
    int nl = 0;
    for (;; ++nl) {
      if (nl == kMgMaxLevels) return false;
      MgLv& L = a.lv[nl];
      const int64_t V = (int64_t)n[0] * n[1] * n[2];
      L.n0 = n[0];
      L.n1 = n[1];
      L.n2 = n[2];
      L.V = (int)V;
      L.rb = n[0] % 2 == 0 && n[1] % 2 == 0 && n[2] % 2 == 0;
      L.split = V <= kMgSplitSites;
      L.d0 = fast_div((unsigned)n[0]);
      L.d1 = fast_div((unsigned)n[1]);
      L.dh = fast_div((unsigned)n[0] / 2);
      at.push_back(words);
      words += (size_t)V * (5 + (L.rb ? 3 : 4) * nr);
      if (n[0] < 4 || n[1] < 4 || n[2] < 4 || V <= 64) break;
      for (int d = 0; d < 3; ++d) n[d] /= 2;
    }
    a.nl = nl + 1;
    a.nlg = 0;
    while (a.nlg < a.nl && a.lv[a.nlg].V > (a.nlg + 1 < a.nl ? kMgCtaSites : kMgCtaLast)) ++a.nlg;
    size_t sites = 0;
    for (int l = a.nlg; l < a.nl; ++l) sites += (size_t)a.lv[l].V;
    if (sites > (size_t)kMgCtaLast || a.nl - a.nlg > kMgCtaLevels) return false;
    smem = 9 * sites * sizeof(double);
    const size_t head = (sizeof(MgOut) + 64) / sizeof(double) + 1;  // result, barrier count
    const size_t parts = (size_t)kMgSlots * kMgQ * std::min<int64_t>(kSumWarps, (m.V + 31) / 32);
    const size_t total = head + parts + words + (size_t)(x ? nr : nr + 1) * m.V;
    block = (double*)memd_dalloc(c, total * sizeof(double));
    if (!block) return false;
    a.out = (MgOut*)block;
    a.arrivals = (unsigned*)((char*)block + ((sizeof(MgOut) + 31) / 32) * 32);
    zero_bytes = head * sizeof(double);
    a.part = block + head;
    double* base = a.part + parts;
    for (int l = 0; l < a.nl; ++l) {
      MgLv& L = a.lv[l];
      double* b = base + at[l];
      const size_t V = (size_t)L.V;
      L.w = b;
      L.dg = b + 3 * V;
      L.idg = b + 4 * V;
      L.f = b + 5 * V;
      L.r = L.f + nr * V;
      L.phi = L.r + nr * V;
      L.alt = L.rb ? nullptr : L.phi + nr * V;
    }
    a.p = base + words;
    a.q = a.lv[0].r;
    a.x = x ? x : a.p + (size_t)nr * m.V;
    a.inv_a = 1.0 / m.a;
    a.inv_a2 = 1.0 / (m.a * m.a);
    a.ie64 = c->ie64;
    return true;
  }
  // clears the barrier count, launches, waits, and reads the result
  template <int NR, int MODE>
  memd_status run(memd_ctx* c, MgOut& h) {
    const cudaStream_t st = c->stream;
    if (cudaMemsetAsync(block, 0, zero_bytes, st) != cudaSuccess ||
        launch_solve<NR, MODE>(a, grid, smem, st) != cudaSuccess ||
        cudaMemcpyAsync(&h, a.out, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return MEMD_ERR_CUDA;
    if (h.timeout) return MEMD_ERR_TIMEOUT;
    return h.converged ? MEMD_OK : MEMD_ERR_RELAX_NOCONV;
  }
};

}  // namespace

// Cell problems: psi_d (3V, stored), and eps_eff[e][d] = mean over links of
// eps_e (delta_ed - grad_e psi_d) (row e, column d).
memd_status mg_eps_eff(memd_ctx* c, double* psi, double eps_eff[9], double tol, int maxit) {
  MgPlan plan;
  if (!plan.build(c, 3, psi)) return MEMD_ERR_OOM;
  plan.a.tol = tol;
  plan.a.maxit = maxit < 400 ? maxit : 400;
  MgOut h;
  const memd_status s = plan.run<3, kMgCells>(c, h);
  if (s == MEMD_OK)
    for (int t = 0; t < 9; ++t) eps_eff[t] = h.sum[t] / (double)c->mesh.V;
  memd_dfree(c, plan.block);
  return s;
}

// D64 (div D = rho, mean M) -> the relaxed field with the same divergence
// and mean: D = -eps grad phi + sum_d E0_d eps (e_d - grad psi_d),
// L phi = div D64, E0 = eps_eff^-1 (M - mean(-eps grad phi)).
memd_status mg_relax(memd_ctx* c, double* D64, const double* psi, const double eps_eff_inv[9],
                     double tol, int maxit, int* iters) {
  MgPlan plan;
  if (!plan.build(c, 1, nullptr)) return MEMD_ERR_OOM;
  plan.a.D64 = D64;
  plan.a.tol = tol;
  plan.a.maxit = maxit < 400 ? maxit : 400;
  MgOut h;
  const memd_status s = plan.run<1, kMgRelax>(c, h);
  if (iters) *iters = s == MEMD_OK ? h.iters : 0;
  const MgLv L = plan.a.lv[0];
  memd_dfree(c, plan.block);
  if (s != MEMD_OK) return s;
  double dm[3], E0[3];
  for (int e = 0; e < 3; ++e) dm[e] = (h.sum[e] - h.sum[3 + e]) / (double)c->mesh.V;
  for (int e = 0; e < 3; ++e)
    E0[e] = eps_eff_inv[3 * e] * dm[0] + eps_eff_inv[3 * e + 1] * dm[1] +
            eps_eff_inv[3 * e + 2] * dm[2];
  if (E0[0] != 0.0 || E0[1] != 0.0 || E0[2] != 0.0)
    k_mg_mean_field<<<(unsigned)((L.V + 255) / 256), 256, 0, c->stream>>>(
        L, c->ie64, psi, MgE0{{E0[0], E0[1], E0[2]}}, plan.a.inv_a, D64);
  return cudaGetLastError() == cudaSuccess ? MEMD_OK : MEMD_ERR_CUDA;
}

}  // namespace memd
