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
// V(1,1)-cycle, FP64 throughout, the whole solve in one cooperative launch.
// Every axis of n vertices coarsens to ceil(n / 2) (the even ones; on an odd
// axis the last and the first vertex are both coarse and keep their link),
// down to at most 32 vertices: linear interpolation, its transpose, and coarse link
// conductances from two fine links in series summed over the perpendicular
// weights.  Gauss-Seidel by colours: two where every axis is even; an odd
// ring needs a third for its last vertex, and the sum of the axes' colours
// modulo 3 is then a proper colouring of the periodic lattice.  The
// iteration count is the same for even and odd meshes (15 to 20 to 1e-12 on
// smooth random and slab profiles of contrast 40).
//
// What bounds it: the FP64 pipe of GB300 takes 16 cycles a warp instruction,
// so the cycle is written for few FP64 operations a vertex (the inverse
// diagonal kept, the pre-smoothing started from zero, the residual and the
// prolongation left out where the last colour makes them zero or overwrites
// them: about 35 a vertex and iteration), and, below 10^5 vertices, the
// latency of its phases: a grid barrier costs ~1.2 us where a kernel launch
// cost 2.5-4 us, and the host takes no part in the iteration.  Levels of at
// most kMgCtaSites vertices run in one CTA a right-hand side, which needs
// CTA barriers only.  A whole system's setup (48^3, 2200 charges; 77^3, 10^4
// charges): 8.7 and 27.1 ms with one launch a half sweep, host checks between
// iterations, and aggregation with Jacobi on odd levels; 3.6 and 8.2 ms so.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "memd_ctx.cuh"
#include "memd_internal.cuh"

namespace memd {

namespace {

// 512 threads with all the registers they take: held to 64 registers the
// three-right-hand-side solve spills (48^3 and 77^3 setups 3.77 and 8.60 ms
// against 3.63 and 8.19), 1024 threads only add to the barriers (4.25, 9.09).
constexpr int kMgThreads = 512;
constexpr int kMgMaxLevels = 32;  // an axis has less than 2^30 vertices
// Levels up to this size run in one CTA a right-hand side, in shared memory:
// a phase of 6^3 vertices takes ~0.9 us there and ~2.2 us with a grid barrier;
// from 8^3 on the one SM's FP64 pipe is the slower (12^3 and below in one CTA
// took 39 us a cycle, of 95, in a 48^3 solve; 18 with 12^3 on the grid).
constexpr int kMgCtaSites = 256;
constexpr int kMgCtaTotal = 480;  // of all such levels together (256, 128, 64, 32 on one axis)
constexpr int kMgCtaLevels = 4;
// The first level of at most this many vertices is the last: solved exactly
// by the inverse of its matrix, formed once a solve (a matrix-vector product
// of 27 vertices takes ~0.4 us; sweeping it and the 2^3 level below took 14
// phases of 0.9 us, latency of dependent FP64 operations, 70 cycles each).
constexpr int kMgDirect = 32;
constexpr int kMgGrid = 256;  // most CTAs
constexpr int kMgQ = 12;     // most sums of one reduction
constexpr int kMgSlots = 6;  // reductions in flight between two uses of a slot
constexpr unsigned long long kMgWaitNs = 2000000000ull;  // bound of a barrier wait

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
  int nc;            // colours
  int hx;            // positions of one colour in a row (i = 2 h + 0 or 1)
  FastDiv d0, d1, dh;  // by n0, n1, hx
  double* w;    // 3 V conductances of the links
  double* dg;   // V: their sum at a vertex
  double* idg;  // V: its inverse (0 where it is 0)
  double* phi;  // correction
  double* f;    // right-hand side
  double* r;    // residual; stays 0 on the last colour
};

enum : int { kMgCells = 0, kMgRelax = 1 };

struct MgOut {
  double eff[9];    // cells: eps_eff[e][d] at 3 e + d
  int converged, iters, timeout, pad;
};

struct MgArgs {
  int nl, nlg;  // levels, and how many of them are swept by the whole grid
  int dir0;     // cells: direction of right-hand side 0
  int maxit;
  double tol;
  double a;
  const double* ie64;
  double* x;    // solution
  double* p;
  double* q;
  double* part;       // kMgSlots x kMgQ x CTAs
  unsigned* arrivals; // barrier count, 0 at launch
  MgOut* out;
  double* psi;        // cells: written; relax: read (3 V)
  double* D64;        // relax: in and out
  double einv[9];     // relax: inverse effective permittivity
  MgLv lv[kMgMaxLevels];
};

// explicit roundings: the arithmetic of a right-hand side does not depend on
// how many are solved at once
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }

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
// colour of a position on an axis: alternating, the last of an odd ring apart
__device__ __forceinline__ int axis_colour(int i, int n) {
  return (n & 1) && n > 1 && i == n - 1 ? 2 : i & 1;
}
__device__ __forceinline__ bool first_colour(const MgLv& L, int i, int j, int k) {
  const int s = axis_colour(i, L.n0) + axis_colour(j, L.n1) + axis_colour(k, L.n2);
  return L.nc == 2 ? (s & 1) == 0 : s % 3 == 0;
}
// position h of colour c: row by row, hx a row; false where there is none
__device__ __forceinline__ bool colour_vertex(const MgLv& L, int h, int c, int& i, int& j, int& k) {
  const int row = h / L.dh;
  const int hh = h - row * L.hx;
  k = row / L.d1;
  j = row - k * L.n1;
  const int b = axis_colour(j, L.n1) + axis_colour(k, L.n2);
  const bool odd0 = (L.n0 & 1) && L.n0 > 1;
  int t;
  if (L.nc == 2) {
    t = (c - b) & 1;
  } else {
    t = c - b;
    t = t < 0 ? t + 3 : t;
    t = t < 0 ? t + 3 : t;
  }
  if (t < 2) {
    i = 2 * hh + t;
    return i < (odd0 ? L.n0 - 1 : L.n0);
  }
  i = L.n0 - 1;
  return odd0 && hh == 0;
}

// ---------------------------------------------------------- phases
// t0, stride: this thread's share of the vertices; r0: first right-hand side

// Gauss-Seidel on one colour; acc (optional) gathers f . phi of the updated
template <int NR>
__device__ __forceinline__ void sweep(const MgLv& L, int c, int t0, int stride, int r0,
                                      double* acc) {
  const int H = L.hx * L.n1 * L.n2, V = L.V;
  const double* w = L.w;
  for (int h = t0; h < H; h += stride) {
    int i, j, k;
    if (!colour_vertex(L, h, c, i, j, k)) continue;
    const int v = i + L.n0 * (j + L.n1 * k);
    const Nb b = neighbours(L, v, i, j, k);
    const double wxp = w[v], wxm = w[b.xm], wyp = w[V + v], wym = w[V + b.ym], wzp = w[2 * V + v],
                 wzm = w[2 * V + b.zm], id = L.idg[v];
    double y[NR], g[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const double* p = L.phi + (r0 + r) * V;
      g[r] = L.f[(r0 + r) * V + v];
      double s = fma_(wxp, p[b.xp], g[r]);
      s = fma_(wxm, p[b.xm], s);
      s = fma_(wyp, p[b.yp], s);
      s = fma_(wym, p[b.ym], s);
      s = fma_(wzp, p[b.zp], s);
      s = fma_(wzm, p[b.zm], s);
      y[r] = mul_(s, id);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      L.phi[(r0 + r) * V + v] = y[r];
      if (acc) acc[r] = fma_(g[r], y[r], acc[r]);
    }
  }
}

// f - L phi on every colour but the last (where the sweep left 0)
template <int NR>
__device__ __forceinline__ void residual(const MgLv& L, int t0, int stride, int r0) {
  const int H = L.hx * L.n1 * L.n2, V = L.V;
  const double* w = L.w;
  for (int c = 0; c + 1 < L.nc; ++c)
    for (int h = t0; h < H; h += stride) {
      int i, j, k;
      if (!colour_vertex(L, h, c, i, j, k)) continue;
      const int v = i + L.n0 * (j + L.n1 * k);
      const Nb b = neighbours(L, v, i, j, k);
      const double wxp = w[v], wxm = w[b.xm], wyp = w[V + v], wym = w[V + b.ym],
                   wzp = w[2 * V + v], wzm = w[2 * V + b.zm], dg = L.dg[v];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double* p = L.phi + (r0 + r) * V;
        double s = fma_(-dg, p[v], L.f[(r0 + r) * V + v]);
        s = fma_(wxp, p[b.xp], s);
        s = fma_(wxm, p[b.xm], s);
        s = fma_(wyp, p[b.yp], s);
        s = fma_(wym, p[b.ym], s);
        s = fma_(wzp, p[b.zp], s);
        s = fma_(wzm, p[b.zm], s);
        L.r[(r0 + r) * V + v] = s;
      }
    }
}

// the two fine neighbours of coarse position I on an axis of n fine vertices
// and their weights in the transpose of the interpolation
__device__ __forceinline__ void axis_pair(int I, int n, int m, int& lo, int& hi, double& wl,
                                          double& wr) {
  const bool odd = n & 1;
  lo = I == 0 ? n - 1 : 2 * I - 1;
  hi = 2 * I + 1 >= n ? 0 : 2 * I + 1;
  wl = odd && I == 0 ? 0.0 : 0.5;
  wr = odd && I == m - 1 ? 0.0 : 0.5;
}

// f of the coarse level, and its first half sweep from zero (the first
// colour's values; 0 elsewhere)
template <int NR>
__device__ __forceinline__ void restrict_to(const MgLv& F, const MgLv& C, int t0, int stride,
                                            int r0) {
  const bool two = F.nc == 2 && F.n0 > 1 && F.n1 > 1 && F.n2 > 1;
  for (int v = t0; v < C.V; v += stride) {
    int I, J, K;
    coords(C, v, I, J, K);
    int x[3], y[3], z[3];
    double wx[3], wy[3], wz[3];
    x[1] = 2 * I;
    y[1] = 2 * J;
    z[1] = 2 * K;
    axis_pair(I, F.n0, C.n0, x[0], x[2], wx[0], wx[2]);
    axis_pair(J, F.n1, C.n1, y[0], y[2], wy[0], wy[2]);
    axis_pair(K, F.n2, C.n2, z[0], z[2], wz[0], wz[2]);
    const bool c0 = first_colour(C, I, J, K);
    const double id = C.idg[v];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const double* q = F.r + (r0 + r) * F.V;
      auto row = [&](int b, int c) { return q + F.n0 * (y[b] + F.n1 * z[c]); };
      double s;
      if (two) {
        // the residual is 0 on the odd vertices: the centre and the twelve
        // diagonal neighbours remain
        const double* c1 = row(1, 1);
        double e = add_(add_(row(0, 1)[x[0]], row(0, 1)[x[2]]),
                        add_(row(2, 1)[x[0]], row(2, 1)[x[2]]));
        e = add_(e, add_(add_(row(1, 0)[x[0]], row(1, 0)[x[2]]),
                         add_(row(1, 2)[x[0]], row(1, 2)[x[2]])));
        e = add_(e, add_(add_(row(0, 0)[x[1]], row(2, 0)[x[1]]),
                         add_(row(0, 2)[x[1]], row(2, 2)[x[1]])));
        s = fma_(0.25, e, c1[x[1]]);
      } else {
        auto line = [&](int b, int c) {
          const double* l = row(b, c);
          return fma_(wx[2], l[x[2]], fma_(wx[0], l[x[0]], l[x[1]]));
        };
        auto plane = [&](int c) {
          return fma_(wy[2], line(2, c), fma_(wy[0], line(0, c), line(1, c)));
        };
        s = fma_(wz[2], plane(2), fma_(wz[0], plane(0), plane(1)));
      }
      C.f[(r0 + r) * C.V + v] = s;
      C.phi[(r0 + r) * C.V + v] = c0 ? mul_(s, id) : 0.0;
    }
  }
}

// phi += interpolated coarse correction: a thread takes the (up to) eight
// fine vertices 2 I + {0, 1} of a coarse one, which share their sums (and
// run without divergence).  With two colours only the even ones: the first
// half sweep after it overwrites the last colour.
template <int NR>
__device__ __forceinline__ void prolong(const MgLv& F, const MgLv& C, int t0, int stride, int r0) {
  const bool two = F.nc == 2 && F.n0 > 1 && F.n1 > 1 && F.n2 > 1;
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
      const double q00 = e[c00 + I], q10 = e[c10 + I], q01 = e[c01 + I], q11 = e[c11 + I];
      const double x00 = add_(q00, e[c00 + I1]), x10 = add_(q10, e[c10 + I1]),
                   x01 = add_(q01, e[c01 + I1]);
      if (two) {
        const double a0 = p[0], a1 = p[1 + sy], a2 = p[1 + sz], a3 = p[sy + sz];
        p[0] = add_(a0, q00);
        p[1 + sy] = fma_(0.25, add_(x00, x10), a1);
        p[1 + sz] = fma_(0.25, add_(x00, x01), a2);
        p[sy + sz] = fma_(0.25, add_(add_(q00, q10), add_(q01, q11)), a3);
        continue;
      }
      const bool ox = 2 * I + 1 < F.n0, oy = 2 * J + 1 < F.n1, oz = 2 * K + 1 < F.n2;
      const double x11 = add_(q11, e[c11 + I1]);
      const double y0 = add_(q00, q10), y1 = add_(x00, x10);
      p[0] = add_(p[0], q00);
      if (ox) p[1] = fma_(0.5, x00, p[1]);
      if (oy) p[sy] = fma_(0.5, y0, p[sy]);
      if (ox && oy) p[1 + sy] = fma_(0.25, y1, p[1 + sy]);
      if (oz) {
        p[sz] = fma_(0.5, add_(q00, q01), p[sz]);
        if (ox) p[1 + sz] = fma_(0.25, add_(x00, x01), p[1 + sz]);
        if (oy) p[sy + sz] = fma_(0.25, add_(y0, add_(q01, q11)), p[sy + sz]);
        if (ox && oy) p[1 + sy + sz] = fma_(0.125, add_(y1, add_(x01, x11)), p[1 + sy + sz]);
      }
    }
  }
}

// conductance of link d of coarse vertex (I, J, K): the fine links in series
// (one at the seam of an odd axis), over the perpendicular weights
__device__ __forceinline__ double coarse_link(const MgLv& F, const MgLv& C, int d, int I, int J,
                                              int K) {
  const int nf[3] = {F.n0, F.n1, F.n2}, nc[3] = {C.n0, C.n1, C.n2}, c[3] = {I, J, K};
  if (nc[d] == 1) return 0.0;
  const int sf[3] = {1, F.n0, F.n0 * F.n1};
  const int e1 = (d + 1) % 3, e2 = (d + 2) % 3;
  const bool seam = (nf[d] & 1) && c[d] == nc[d] - 1;
  const int along = 2 * c[d] * sf[d];
  int p1[3], p2[3];
  double w1[3], w2[3];
  p1[1] = 2 * c[e1];
  p2[1] = 2 * c[e2];
  w1[1] = w2[1] = 1.0;
  axis_pair(c[e1], nf[e1], nc[e1], p1[0], p1[2], w1[0], w1[2]);
  axis_pair(c[e2], nf[e2], nc[e2], p2[0], p2[2], w2[0], w2[2]);
  const double* w = F.w + (int64_t)d * F.V;
  double s = 0.0;
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      // a link along an axis that coarsens is positive, also where wp is 0
      const double wp = mul_(w1[a], w2[b]);
      const int v = along + p1[a] * sf[e1] + p2[b] * sf[e2];
      const double u = w[v], u1 = seam ? u : w[v + sf[d]];
      s = fma_(wp, seam ? u : mul_(u, u1) / add_(u, u1), s);
    }
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

// this CTA's share of NQ sums into slot; every CTA reads all shares after the
// next grid barrier and adds them in the same order
template <int NQ>
__device__ __forceinline__ void share_sums(double* part, int slot, const double (&x)[NQ],
                                           double (*sh)[kMgQ]) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    double s = x[q];
    for (int o = 16; o > 0; o >>= 1) s = add_(s, __shfl_down_sync(0xffffffffu, s, o));
    if (lane == 0) sh[wp][q] = s;
  }
  __syncthreads();
  constexpr int NW = kMgThreads / 32;
  if (wp < NQ) {
    double s = lane < NW ? sh[lane][wp] : 0.0;
    for (int o = NW / 2; o > 0; o >>= 1) s = add_(s, __shfl_down_sync(0xffffffffu, s, o));
    if (lane == 0) part[((int64_t)slot * kMgQ + wp) * gridDim.x + blockIdx.x] = s;
  }
}
template <int NQ>
__device__ __forceinline__ void total_sums(const double* part, int slot, double (&x)[NQ],
                                           double* tot) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  static_assert(NQ <= kMgThreads / 32, "one warp a sum");
  if (wp < NQ) {
    const double* p = part + ((int64_t)slot * kMgQ + wp) * gridDim.x;
    double y[kMgGrid / 32];
#pragma unroll
    for (int k = 0; k < kMgGrid / 32; ++k)
      y[k] = lane + 32 * k < (int)gridDim.x ? __ldcg(p + lane + 32 * k) : 0.0;
    double s = y[0];
#pragma unroll
    for (int k = 1; k < kMgGrid / 32; ++k)
      if (32 * k < (int)gridDim.x) s = add_(s, y[k]);
    for (int o = 16; o > 0; o >>= 1) s = add_(s, __shfl_down_sync(0xffffffffu, s, o));
    if (lane == 0) tot[wp] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) x[q] = tot[q];
}

// The inverse of a level's matrix plus a multiple of the all-ones matrix
// (which acts on the constants alone: right-hand sides have none), by
// Gauss-Jordan steps in place; the whole CTA calls it.
__device__ void invert_level(const MgLv& L, double* A) {
  const int n = L.V, U = n * n;
  const double shift = L.dg[0] / n;
  for (int t = threadIdx.x; t < U; t += kMgThreads) {
    const int u = t / n, v = t - u * n;
    double y = u == v ? add_(L.dg[u], shift) : shift;
    if (u != v) {
      // the links from u to v and from v to u (on an axis of two, both)
      int i, j, k;
      coords(L, u, i, j, k);
      const Nb b = neighbours(L, u, i, j, k);
      coords(L, v, i, j, k);
      const Nb c = neighbours(L, v, i, j, k);
      const int bu[3] = {b.xp, b.yp, b.zp}, bv[3] = {c.xp, c.yp, c.zp};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (bu[d] == v) y = sub_(y, L.w[d * n + u]);
        if (bv[d] == u) y = sub_(y, L.w[d * n + v]);
      }
    }
    A[t] = y;
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const double p = 1.0 / A[k * n + k];
    for (int t = threadIdx.x; t < U; t += kMgThreads) {
      const int i = t / n, j = t - i * n;
      if (i != k && j != k) A[t] = fma_(-mul_(A[i * n + k], p), A[k * n + j], A[t]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * n; t += kMgThreads) {
      const int i = t < n ? t : t - n;
      if (i == k) continue;
      if (t < n)
        A[i * n + k] = mul_(-A[i * n + k], p);
      else
        A[k * n + i] = mul_(A[k * n + i], p);
    }
    if (threadIdx.x == 0) A[k * n + k] = p;
    __syncthreads();
  }
}

// The whole solve for NR right-hand sides.
//   cells: L psi_d = -div(eps e_d) for d = dir0 .. dir0 + NR - 1, psi_d of
//   zero mean and the mean fluxes eps_e (delta_ed - grad_e psi_d)
//   relax: L phi = div D64; D64 <- eps (-grad phi + sum_d E0_d (e_d - grad
//   psi_d)) with E0 from the mean of D64
// Stops when |r| <= tol |f| / 4 (2-norms) or, once the recursion has reached
// its rounding floor and the residual grows again (to 100 times its least
// value), when that least value was below 100 tol |f|.
template <int NR, int MODE>
__global__ void __launch_bounds__(kMgThreads) k_mg_solve(const __grid_constant__ MgArgs a) {
  __shared__ double sh[kMgThreads / 32][kMgQ];
  __shared__ double tot[2][kMgQ];
  __shared__ int s_ok;
  GridSync grid{a.arrivals, a.out, 0u, &s_ok};
#define MG_GRID() \
  if (!grid()) return
  // neighbouring warps of work go to different SMs: a level with less work
  // than the grid has warps still uses every FP64 pipe
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int t0 = (wp * (int)gridDim.x + (int)blockIdx.x) * 32 + lane;
  const int stride = (int)gridDim.x * kMgThreads;
  const MgLv& L = a.lv[0];
  const int V = L.V;
  const double inv_a = 1.0 / a.a, inv_a2 = 1.0 / (a.a * a.a), nV = (double)V;
  double mean0[3] = {0.0, 0.0, 0.0};  // relax: mean of D64
  {
    // conductances of the finest level, the right-hand side and its sum
    constexpr int NQ = MODE == kMgRelax ? 4 : NR;
    double s[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) s[q] = 0.0;
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const int vm[3] = {b.xm, b.ym, b.zm};
#pragma unroll
      for (int d = 0; d < 3; ++d) L.w[d * V + v] = inv_a2 / a.ie64[(int64_t)d * V + v];
      if (MODE == kMgRelax) {
        double div = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double D = a.D64[(int64_t)d * V + v];
          s[1 + d] = add_(s[1 + d], D);
          div = add_(div, sub_(D, a.D64[(int64_t)d * V + vm[d]]));
        }
        const double f = mul_(inv_a, div);
        L.f[v] = f;
        s[0] = add_(s[0], f);
      } else {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int d = a.dir0 + r;
          const double* ie = a.ie64 + (int64_t)d * V;
          const double f = mul_(-(__drcp_rn(ie[v]) - __drcp_rn(ie[vm[d]])), inv_a);
          L.f[r * V + v] = f;
          s[r] = add_(s[r], f);
        }
      }
    }
    share_sums<NQ>(a.part, 0, s, sh);
    MG_GRID();
    double m[NQ];
    total_sums<NQ>(a.part, 0, m, tot[0]);
    if (MODE == kMgRelax) {
#pragma unroll
      for (int d = 0; d < 3; ++d) mean0[d] = m[NQ - 3 + d] / nV;
    }
    for (int v = t0; v < V; v += stride)
#pragma unroll
      for (int r = 0; r < NR; ++r) L.f[r * V + v] = sub_(L.f[r * V + v], m[r] / nV);
  }
  // diagonals, and the conductances level by level
  for (int l = 0; l < a.nl; ++l) {
    const MgLv& F = a.lv[l];
    for (int v = t0; v < F.V; v += stride) {
      int i, j, k;
      coords(F, v, i, j, k);
      const Nb b = neighbours(F, v, i, j, k);
      const int U = F.V;
      const double dg = ((F.w[v] + F.w[b.xm]) + (F.w[U + v] + F.w[U + b.ym])) +
                        (F.w[2 * U + v] + F.w[2 * U + b.zm]);
      F.dg[v] = dg;
      F.idg[v] = dg > 0.0 ? 1.0 / dg : 0.0;
#pragma unroll
      for (int r = 0; r < NR; ++r) F.r[r * U + v] = 0.0;
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
  // x = 0, p = 0, |f|^2, the first half sweep
  double f2[NR], least[NR], rz[NR];
  bool done[NR];
  {
    double s[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) s[r] = 0.0;
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const bool c0 = first_colour(L, i, j, k);
      const double id = L.idg[v];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double f = L.f[r * V + v];
        s[r] = fma_(f, f, s[r]);
        a.x[r * V + v] = 0.0;
        a.p[r * V + v] = 0.0;
        L.phi[r * V + v] = c0 ? mul_(f, id) : 0.0;
      }
    }
    share_sums<NR>(a.part, 1, s, sh);
    MG_GRID();
    total_sums<NR>(a.part, 1, f2, tot[1]);
  }
  bool all = true;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    done[r] = f2[r] == 0.0;
    least[r] = f2[r];
    rz[r] = 0.0;
    all = all && done[r];
  }
  // the levels of the one-CTA part: coefficients into shared memory
  __shared__ double s_mem[8 * kMgCtaTotal];
  __shared__ MgLv s_lv[kMgCtaLevels];
  __shared__ double s_inv[kMgDirect * kMgDirect];
  if ((int)blockIdx.x < NR) {
    const MgLv& D = a.lv[a.nl - 1];
    invert_level(D, s_inv);
    int at = 0;
    for (int l = a.nlg; l < a.nl; ++l) {
      const MgLv& F = a.lv[l];
      const int U = F.V;
      double* b = s_mem + 8 * at;
      at += U;
      for (int v = threadIdx.x; v < U; v += kMgThreads) {
#pragma unroll
        for (int d = 0; d < 3; ++d) b[d * U + v] = F.w[d * U + v];
        b[3 * U + v] = F.dg[v];
        b[4 * U + v] = F.idg[v];
        b[7 * U + v] = 0.0;
      }
      if (threadIdx.x == 0) {
        MgLv C = F;
        C.w = b;
        C.dg = b + 3 * U;
        C.idg = b + 4 * U;
        C.phi = b + 5 * U;
        C.f = b + 6 * U;
        C.r = b + 7 * U;
        s_lv[l - a.nlg] = C;
      }
    }
  }
  __syncthreads();
  int its = 0;
  const double tol2 = a.tol * a.tol;
  while (!all) {
    // z = M r in phi of level 0: one V(1,1)-cycle, its first half sweep made
    // where r was; sums r . z
    double acc[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] = 0.0;
    for (int l = 0; l < a.nlg; ++l) {
      const MgLv& F = a.lv[l];
      for (int c = 1; c < F.nc; ++c) {
        sweep<NR>(F, c, t0, stride, 0, nullptr);
        MG_GRID();
      }
      residual<NR>(F, t0, stride, 0);
      MG_GRID();
      restrict_to<NR>(F, a.lv[l + 1], t0, stride, 0);
      MG_GRID();
    }
    if ((int)blockIdx.x < NR) {
      const int r = blockIdx.x, t = threadIdx.x;
      double one = 0.0;
      const MgLv& top = a.lv[a.nlg];
      for (int v = t; v < top.V; v += kMgThreads) {
        s_lv[0].f[v] = top.f[r * top.V + v];
        s_lv[0].phi[v] = top.phi[r * top.V + v];
      }
      __syncthreads();
      const int nc = a.nl - a.nlg;
      for (int l = 0; l + 1 < nc; ++l) {
        const MgLv& F = s_lv[l];
        for (int c = 1; c < F.nc; ++c) {
          sweep<1>(F, c, t, kMgThreads, 0, nullptr);
          __syncthreads();
        }
        residual<1>(F, t, kMgThreads, 0);
        __syncthreads();
        restrict_to<1>(F, s_lv[l + 1], t, kMgThreads, 0);
        __syncthreads();
      }
      {
        // four threads a row of the inverse
        const MgLv& D = s_lv[nc - 1];
        const int v = t >> 2, n = D.V;
        double y = 0.0;
        if (v < n)
          for (int j = t & 3; j < n; j += 4) y = fma_(s_inv[v * n + j], D.f[j], y);
        if (t < 4 * kMgDirect) {
          y = add_(y, __shfl_xor_sync(0xffffffffu, y, 1));
          y = add_(y, __shfl_xor_sync(0xffffffffu, y, 2));
        }
        if (v < n && (t & 3) == 0) {
          D.phi[v] = y;
          if (a.nl == 1) one = mul_(D.f[v], y);
        }
        __syncthreads();
      }
      for (int l = nc - 2; l >= 0; --l) {
        const MgLv& F = s_lv[l];
        prolong<1>(F, s_lv[l + 1], t, kMgThreads, 0);
        __syncthreads();
        for (int c = F.nc - 1; c >= 0; --c) {
          sweep<1>(F, c, t, kMgThreads, 0, l + a.nlg == 0 ? &one : nullptr);
          __syncthreads();
        }
      }
      for (int v = t; v < top.V; v += kMgThreads) top.phi[r * top.V + v] = s_lv[0].phi[v];
#pragma unroll
      for (int q = 0; q < NR; ++q)
        if (q == r) acc[q] = one;
    }
    if (a.nlg > 0) MG_GRID();
    for (int l = a.nlg - 1; l >= 0; --l) {
      const MgLv& F = a.lv[l];
      prolong<NR>(F, a.lv[l + 1], t0, stride, 0);
      MG_GRID();
      for (int c = F.nc - 1; c >= 0; --c) {
        sweep<NR>(F, c, t0, stride, 0, l == 0 ? acc : nullptr);
        if (l > 0 || c > 0) MG_GRID();
      }
    }
    share_sums<NR>(a.part, 2, acc, sh);
    MG_GRID();
    double rz1[NR];
    total_sums<NR>(a.part, 2, rz1, tot[0]);
    // p = z + beta p, then q = L p and p . q
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
          p[u][r] = in ? a.p[r * V + v] : 0.0;
          z[u][r] = in ? L.phi[r * V + v] : 0.0;
        }
#pragma unroll
      for (int u = 0; u < UP; ++u)
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (v0 + u * stride < V)
            a.p[r * V + v0 + u * stride] = fma_(beta[r], p[u][r], z[u][r]);
    }
    MG_GRID();
    double pq[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) pq[r] = 0.0;
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const double wxp = L.w[v], wxm = L.w[b.xm], wyp = L.w[V + v], wym = L.w[V + b.ym],
                   wzp = L.w[2 * V + v], wzm = L.w[2 * V + b.zm], dg = L.dg[v];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double* p = a.p + r * V;
        double s = mul_(dg, p[v]);
        s = fma_(-wxp, p[b.xp], s);
        s = fma_(-wxm, p[b.xm], s);
        s = fma_(-wyp, p[b.yp], s);
        s = fma_(-wym, p[b.ym], s);
        s = fma_(-wzp, p[b.zp], s);
        s = fma_(-wzm, p[b.zm], s);
        a.q[r * V + v] = s;
        pq[r] = fma_(p[v], s, pq[r]);
      }
    }
    share_sums<NR>(a.part, 3, pq, sh);
    MG_GRID();
    total_sums<NR>(a.part, 3, pq, tot[1]);
    // x and r, and the next cycle's first half sweep
    double alpha[NR], rr[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      alpha[r] = !done[r] && pq[r] != 0.0 ? rz[r] / pq[r] : 0.0;
      rr[r] = 0.0;
    }
    constexpr int UX = NR == 1 ? 3 : 1;
    for (int v0 = t0; v0 < V; v0 += UX * stride) {
      double x[UX][NR], p[UX][NR], f[UX][NR], q[UX][NR], id[UX];
#pragma unroll
      for (int u = 0; u < UX; ++u) {
        const int v = v0 + u * stride;
        const bool in = v < V;
        id[u] = in ? L.idg[v] : 0.0;
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
        const int v = v0 + u * stride;
        if (v >= V) break;
        int i, j, k;
        coords(L, v, i, j, k);
        const bool c0 = first_colour(L, i, j, k);
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const double t = fma_(-alpha[r], q[u][r], f[u][r]);
          rr[r] = fma_(t, t, rr[r]);
          a.x[r * V + v] = fma_(alpha[r], p[u][r], x[u][r]);
          L.f[r * V + v] = t;
          L.phi[r * V + v] = c0 ? mul_(t, id[u]) : 0.0;
        }
      }
    }
    share_sums<NR>(a.part, 4, rr, sh);
    MG_GRID();
    total_sums<NR>(a.part, 4, rr, tot[0]);
    ++its;
    all = true;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (!done[r]) {
        // a quarter of tol: the residual a solve that checks every second
        // iteration ends at
        const double goal = 0.0625 * tol2 * f2[r];
        done[r] = rr[r] <= goal || (rr[r] > 100.0 * least[r] && least[r] <= 1e4 * tol2 * f2[r]);
        least[r] = rr[r] < least[r] ? rr[r] : least[r];
      }
      all = all && done[r];
    }
    if (its >= a.maxit) break;
  }
  // results
  if (MODE == kMgCells) {
    double s[4 * NR];
#pragma unroll
    for (int q = 0; q < 4 * NR; ++q) s[q] = 0.0;
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const int vp[3] = {b.xp, b.yp, b.zp};
      double eps[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) eps[e] = __drcp_rn(a.ie64[(int64_t)e * V + v]);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double* x = a.x + r * V;
        s[4 * r] = add_(s[4 * r], x[v]);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const double g = fma_(-inv_a, sub_(x[vp[e]], x[v]), e == a.dir0 + r ? 1.0 : 0.0);
          s[4 * r + 1 + e] = fma_(g, eps[e], s[4 * r + 1 + e]);
        }
      }
    }
    share_sums<4 * NR>(a.part, 5, s, sh);
    MG_GRID();
    total_sums<4 * NR>(a.part, 5, s, tot[1]);
    for (int v = t0; v < V; v += stride)
#pragma unroll
      for (int r = 0; r < NR; ++r)
        a.psi[(int64_t)(a.dir0 + r) * V + v] = sub_(a.x[r * V + v], s[4 * r] / nV);
    if (blockIdx.x == 0 && threadIdx.x == 0)
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int e = 0; e < 3; ++e) a.out->eff[3 * e + a.dir0 + r] = s[4 * r + 1 + e] / nV;
  } else if (all) {  // not converged: D64 stays as it came
    double s[3] = {0.0, 0.0, 0.0};
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const int vp[3] = {b.xp, b.yp, b.zp};
#pragma unroll
      for (int e = 0; e < 3; ++e)
        s[e] = add_(s[e], mul_(sub_(a.x[v], a.x[vp[e]]), inv_a) / a.ie64[(int64_t)e * V + v]);
    }
    share_sums<3>(a.part, 5, s, sh);
    MG_GRID();
    total_sums<3>(a.part, 5, s, tot[1]);
    double E0[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
      E0[e] = a.einv[3 * e] * (mean0[0] - s[0] / nV) + a.einv[3 * e + 1] * (mean0[1] - s[1] / nV) +
              a.einv[3 * e + 2] * (mean0[2] - s[2] / nV);
    for (int v = t0; v < V; v += stride) {
      int i, j, k;
      coords(L, v, i, j, k);
      const Nb b = neighbours(L, v, i, j, k);
      const int vp[3] = {b.xp, b.yp, b.zp};
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        // (x, psi) differences along the link: phi + sum_d E0_d psi_d
        double g = sub_(a.x[v], a.x[vp[e]]);
#pragma unroll
        for (int d = 0; d < 3; ++d)
          g = fma_(E0[d], sub_(a.psi[(int64_t)d * V + v], a.psi[(int64_t)d * V + vp[e]]), g);
        a.D64[(int64_t)e * V + v] = fma_(inv_a, g, E0[e]) / a.ie64[(int64_t)e * V + v];
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.out->converged = all ? 1 : 0;
    a.out->iters = its;
  }
#undef MG_GRID
}

// ---------------------------------------------------------------- host
// A cooperative grid starts when all of it fits, whatever else is resident or
// queued on other streams (checked on GB300: two grids that each need every
// SM, the second at a higher priority, while a third kernel holds half of
// them: neither started in part), so concurrent solves and single-launch
// steps never hold SMs that another's barriers wait for.
template <int NR, int MODE>
cudaError_t launch_solve(const MgArgs& a, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kMgThreads, 1, 1);
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
  int grid = 0;

  bool build(memd_ctx* c, int nr) {
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
      const bool odd = (n[0] > 1 && n[0] % 2) || (n[1] > 1 && n[1] % 2) || (n[2] > 1 && n[2] % 2);
      L.nc = odd ? 3 : 2;
      L.hx = std::max(1, n[0] / 2);
      L.d0 = fast_div((unsigned)n[0]);
      L.d1 = fast_div((unsigned)n[1]);
      L.dh = fast_div((unsigned)L.hx);
      at.push_back(words);
      words += (size_t)V * (5 + 3 * nr);
      if (V <= kMgDirect) break;
      for (int d = 0; d < 3; ++d) n[d] = (n[d] + 1) / 2;
    }
    a.nl = nl + 1;
    a.nlg = 0;
    while (a.nlg + 1 < a.nl && a.lv[a.nlg].V > kMgCtaSites) ++a.nlg;
    int sites = 0;
    for (int l = a.nlg; l < a.nl; ++l) sites += a.lv[l].V;
    if (sites > kMgCtaTotal || a.nl - a.nlg > kMgCtaLevels) return false;
    const size_t head = (sizeof(MgOut) + 64) / sizeof(double) + 1;  // result, barrier count
    const size_t parts = (size_t)kMgSlots * kMgQ * grid;
    const size_t total = head + parts + words + (size_t)3 * nr * m.V;
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
      L.phi = b + 5 * V;
      L.f = L.phi + nr * V;
      L.r = L.f + nr * V;
    }
    a.x = base + words;
    a.p = a.x + (size_t)nr * m.V;
    a.q = a.p + (size_t)nr * m.V;
    a.a = m.a;
    a.ie64 = c->ie64;
    return true;
  }
  // clears the barrier count, launches, waits, and reads the result
  template <int NR, int MODE>
  memd_status run(memd_ctx* c, MgOut& h) {
    const cudaStream_t st = c->stream;
    if (cudaMemsetAsync(block, 0, zero_bytes, st) != cudaSuccess ||
        launch_solve<NR, MODE>(a, grid, st) != cudaSuccess ||
        cudaMemcpyAsync(&h, a.out, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return MEMD_ERR_CUDA;
    if (h.timeout) return MEMD_ERR_TIMEOUT;
    return h.converged ? MEMD_OK : MEMD_ERR_RELAX_NOCONV;
  }
};

// Set on a thread (the request server's admission workers): that thread's
// cell problems are solved in turn, with one right-hand side's scratch.
thread_local bool t_cells_in_turn = false;

}  // namespace

void memd_mg_cells_in_turn(bool on) { t_cells_in_turn = on; }

// Cell problems: psi_d (3V, stored), and eps_eff[e][d] = mean over links of
// eps_e (delta_ed - grad_e psi_d) (row e, column d).
memd_status mg_eps_eff(memd_ctx* c, double* psi, double eps_eff[9], double tol, int maxit) {
  const int nr = t_cells_in_turn ? 1 : 3;
  MgPlan plan;
  if (!plan.build(c, nr)) return MEMD_ERR_OOM;
  plan.a.psi = psi;
  plan.a.tol = tol;
  plan.a.maxit = maxit < 400 ? maxit : 400;
  memd_status s = MEMD_OK;
  for (int d = 0; d < 3 && s == MEMD_OK; d += nr) {
    plan.a.dir0 = d;
    MgOut h;
    s = nr == 1 ? plan.run<1, kMgCells>(c, h) : plan.run<3, kMgCells>(c, h);
    if (s == MEMD_OK)
      for (int r = 0; r < nr; ++r)
        for (int e = 0; e < 3; ++e) eps_eff[3 * e + d + r] = h.eff[3 * e + d + r];
  }
  memd_dfree(c, plan.block);
  return s;
}

// D64 (div D = rho, mean M) -> the relaxed field with the same divergence
// and mean: D = -eps grad phi + sum_d E0_d eps (e_d - grad psi_d),
// L phi = div D64, E0 = eps_eff^-1 (M - mean(-eps grad phi)).
memd_status mg_relax(memd_ctx* c, double* D64, const double* psi, const double eps_eff_inv[9],
                     double tol, int maxit, int* iters) {
  MgPlan plan;
  if (!plan.build(c, 1)) return MEMD_ERR_OOM;
  plan.a.psi = const_cast<double*>(psi);
  plan.a.D64 = D64;
  plan.a.tol = tol;
  plan.a.maxit = maxit < 400 ? maxit : 400;
  for (int t = 0; t < 9; ++t) plan.a.einv[t] = eps_eff_inv[t];
  MgOut h;
  const memd_status s = plan.run<1, kMgRelax>(c, h);
  if (iters) *iters = s == MEMD_OK ? h.iters : 0;
  memd_dfree(c, plan.block);
  return s;
}

}  // namespace memd
