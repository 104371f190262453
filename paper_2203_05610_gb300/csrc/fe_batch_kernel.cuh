// fe_batch_kernel.cuh -- the kernel of fe_batch.cu: many small nonlinear solves in one launch: one CTA solves
// one request from its first residual to convergence, so a batch of up to
// (SMs x CTAs per SM) requests runs as a single kernel with no host round
// trip per iteration.  The solvers are those of nl_solve.cu (arxiv
// 2203.05610, Section "Numerical solvers", Appendix A options):
//   NK / iNK: Newton with GMRES(restart) right-preconditioned by the nodal
//             block-Jacobi, fixed ksp_rtol or the Eisenstat-Walker forcing
//             (choice 1 with the safeguard and the cap), full step;
//   B / iB  : L-BFGS two-loop over the stored pairs with H0 = block-Jacobi
//             of K(d_0) (B) or GMRES on K(d_0) at ksp_rtol (iB), full step.
// Every step is a CTA-level loop over the request's elements, nodes or
// unknowns, with the element bodies of fe_element.cuh; reductions are CTA
// sums in a fixed order, so a request's result does not depend on the
// other requests of its batch.  Residuals, Krylov vectors, the Arnoldi
// orthogonalisation and the L-BFGS inner products are FP64; the tangent,
// its block-Jacobi and the SpMV are in T (float: the mixed form, double:
// FP64 throughout).  Displacement-form meshes with nodal block-Jacobi only
// (no pressure space, AMG, follower faces or inertia).
#pragma once
#include "../../include/fe_batch.h"
#include "fe_element.cuh"

namespace {

constexpr int BATCH_MAX_COLORS = 64;
constexpr int BATCH_HIST = FE_BATCH_HIST;       // history entries and the L-BFGS pair cap
constexpr int BATCH_MAX_RESTART = 100;

}  // namespace

// one request of a batch: its mesh's device arrays, options and workspace
struct BatchReq {
  // mesh
  int nn, ne, ncolors;
  int64_t nnzb;
  const int *conn, *perm, *node_ptr, *node_list, *row_ptr, *col, *emap, *diag_pos;
  const int *ks_ptr, *ks_col, *ks_kpos;
  const double *geo, *X, *fib, *fext1, *ks_val;
  const uint8_t* fixmask;
  MatParams mp;
  double load;
  int cstart[BATCH_MAX_COLORS + 1];
  // solver
  int method, max_it, restart, kmaxit, mcap;
  double tol, ksp_rtol, ksp_atol, ew0, ewmax, dtol;
  // workspace: d (in/out) and the rest
  double *d, *r, *rn, *dl, *t, *w, *zb, *gr, *rel, *V, *S, *Y;
  void *K, *Dinv;
  fe_batch_out* out;
};

// CTA reductions that do not depend on the CTA's shape: 256 virtual lanes,
// lane v summing the terms i = v, v + 256, ... in order, each group of 32
// lanes reduced by the same shuffle tree, the 8 group sums added in order by
// one thread.  A request therefore gets bit-identical results with 128 or
// 256 threads per CTA (the launch shape the autotuner picks).
constexpr int VLANES = 256;
template <class F>
__device__ __forceinline__ double cta_vsum(int64_t n, F f, double* sh8, double* slot) {
  const int lane = threadIdx.x & 31;
  for (int vw = threadIdx.x >> 5; vw < VLANES / 32; vw += blockDim.x >> 5) {
    double s = 0.0;
    for (int64_t i = vw * 32 + lane; i < n; i += VLANES) s += f(i);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) sh8[vw] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < VLANES / 32; k++) t += sh8[k];
    *slot = t;
  }
  __syncthreads();
  const double r = *slot;
  __syncthreads();
  return r;
}

__device__ __forceinline__ double cta_dot(const double* a, const double* b, int64_t n, double* sh8, double* slot) {
  return cta_vsum(n, [&](int64_t i) { return a[i] * b[i]; }, sh8, slot);
}

// y = a x + b y over the CTA (no trailing barrier: callers sync before reading y elsewhere)
__device__ __forceinline__ void cta_axpby(double a, const double* x, double b, double* y, int64_t n) {
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) y[i] = a * x[i] + (b == 0.0 ? 0.0 : b * y[i]);
}

// R(d) into r; returns ||R||
template <int ORDER>
__device__ double cta_residual(const BatchReq& q, const double* d, double* r, double* sh8, double* slot) {
  constexpr int NQ = ORDER == 1 ? 1 : 4;
  constexpr int NEN = ORDER == 1 ? 4 : 10;
  const int nitems = q.ne * NQ;
  for (int base = 0; base < nitems; base += blockDim.x)
    elem_residual_item<ORDER, false>(base + (int)threadIdx.x, q.ne, q.conn, q.geo, d, q.nn, 0, q.mp, q.fib, 0.0,
                                     q.rel, nullptr);
  __syncthreads();
  const FollowerFaces none{0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  for (int a = threadIdx.x; a < q.nn; a += blockDim.x)
    gather_node<ORDER, false>(a, q.nn, NEN, q.node_ptr, q.node_list, q.rel, q.fext1, q.load, q.ks_ptr, q.ks_col,
                              q.ks_val, d, q.fixmask, 0, nullptr, nullptr, nullptr, none, nullptr, r,
                              (int64_t)q.ne * NEN);
  __syncthreads();
  return sqrt(cta_dot(r, r, 3 * (int64_t)q.nn, sh8, slot));
}

// tangent K(d) in T with its block-Jacobi inverse
template <int ORDER, class T>
__device__ void cta_tangent(const BatchReq& q, const double* d) {
  using C = TanCfg<ORDER, T>;
  T* K = (T*)q.K;
  const int64_t nval = ((q.nnzb + 31) / 32) * 288;  // kv_count
  for (int64_t i = threadIdx.x; i < nval; i += blockDim.x) K[i] = T(0);
  __syncthreads();
  for (int c = 0; c < q.ncolors; c++) {
    const int start = q.cstart[c], nel = q.cstart[c + 1] - start;
    const int ntiles = (nel + C::EPB - 1) / C::EPB;
    for (int tile = 0; tile < ntiles; tile++) {
      tangent_tile<ORDER, T>(tile, nel, q.perm + start, q.conn, q.geo, d, q.nn, 0, q.mp, q.fib, q.emap, nullptr,
                             q.fixmask, 0.0, K, nullptr, q.nnzb);
      __syncthreads();
    }
  }
  const FollowerFaces none{0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  for (int a = threadIdx.x; a < q.nn; a += blockDim.x)
    face_blocks_row<ORDER, T>(a, q.nn, q.ks_ptr, q.ks_col, q.ks_val, q.ks_kpos, q.fixmask, none, d, q.load, K);
  __syncthreads();
  for (int a = threadIdx.x; a < q.nn; a += blockDim.x)
    diag_inverse_row<T, T>(a, q.nn, q.diag_pos, q.fixmask, K, (T*)q.Dinv);
  __syncthreads();
}

// z = D^{-1} x (nodal 3x3 blocks, arithmetic in T; z in T where the product
// K z reads it in T anyway)
template <class T, class Z>
__device__ __forceinline__ void cta_pc(const BatchReq& q, const double* __restrict__ x, Z* __restrict__ z) {
  const T* Dv = (const T*)q.Dinv;
  for (int a = threadIdx.x; a < q.nn; a += blockDim.x) {
    const T* D = Dv + (int64_t)a * 9;
    const T x0 = (T)x[3 * (int64_t)a], x1 = (T)x[3 * (int64_t)a + 1], x2 = (T)x[3 * (int64_t)a + 2];
    z[3 * (int64_t)a] = (Z)(D[0] * x0 + D[1] * x1 + D[2] * x2);
    z[3 * (int64_t)a + 1] = (Z)(D[3] * x0 + D[4] * x1 + D[5] * x2);
    z[3 * (int64_t)a + 2] = (Z)(D[6] * x0 + D[7] * x1 + D[8] * x2);
  }
}

// y = K x: LPR lanes per node row (P1 rows have up to 15 blocks, P2 rows 10 to
// 65), so a warp has 32 / LPR rows' chains of loads in flight (a warp per row:
// 14 us for the 243 rows of a Cook 8x8x2 request); arithmetic in A (T, or
// double for the FP64-accumulated products of the EW test)
template <int ORDER, class T, class A, class X, class Y>
__device__ __forceinline__ void cta_spmv(const BatchReq& q, const X* __restrict__ x, Y* __restrict__ y) {
  constexpr int LPR = ORDER == 1 ? 4 : 8;
  const T* __restrict__ K = (const T*)q.K;
  const int sub = threadIdx.x % LPR, grp = threadIdx.x / LPR, ng = blockDim.x / LPR;
  const int rounds = (q.nn + ng - 1) / ng;  // (every lane takes part in the shuffles)
  int p = 0, p1 = 0;
  if (grp < q.nn) {
    p = q.row_ptr[grp];
    p1 = q.row_ptr[grp + 1];
  }
  for (int it = 0; it < rounds; it++) {
    const int a = it * ng + grp, an = a + ng;
    int pn = 0, pn1 = 0;
    if (an < q.nn) {  // the next row's range, ahead of this row's products
      pn = q.row_ptr[an];
      pn1 = q.row_ptr[an + 1];
    }
    A s0 = A(0), s1 = A(0), s2 = A(0);
#pragma unroll 4
    for (int k = p + sub; k < p1; k += LPR) {
      const X* xb = x + 3 * (int64_t)q.col[k];
      const A x0 = (A)xb[0], x1 = (A)xb[1], x2 = (A)xb[2];
      s0 += (A)K[kv_index(k, 0)] * x0 + (A)K[kv_index(k, 1)] * x1 + (A)K[kv_index(k, 2)] * x2;
      s1 += (A)K[kv_index(k, 3)] * x0 + (A)K[kv_index(k, 4)] * x1 + (A)K[kv_index(k, 5)] * x2;
      s2 += (A)K[kv_index(k, 6)] * x0 + (A)K[kv_index(k, 7)] * x1 + (A)K[kv_index(k, 8)] * x2;
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1) {
      s0 += __shfl_down_sync(0xffffffffu, s0, off, LPR);
      s1 += __shfl_down_sync(0xffffffffu, s1, off, LPR);
      s2 += __shfl_down_sync(0xffffffffu, s2, off, LPR);
    }
    if (sub == 0 && a < q.nn) {
      y[3 * (int64_t)a] = (Y)s0;
      y[3 * (int64_t)a + 1] = (Y)s1;
      y[3 * (int64_t)a + 2] = (Y)s2;
    }
    p = pn;
    p1 = pn1;
  }
}

// ---- orthogonalisation of one Arnoldi vector
// Modified Gram-Schmidt over blocks of BLK basis vectors: the products of a
// block with w are taken together and h = T s, T = (I + strictly lower part of
// the block's Gram matrix)^-1, is what subtracting one vector after another
// gives (up to rounding); T grows by a row with each vector, from products
// that ride along with its norm.  w and the block stay in registers, so the
// basis is read once and w not at all in between, and the sums of BLK products
// share their reduction: 9 FP64 additions per warp for 8 sums instead of 40,
// one barrier instead of four.  On GB300 an FP64 instruction holds its quarter
// of the SM for 64 cycles whatever its active lanes, predicated off included,
// so the count of instructions is the time: the values per lane (KV) and the
// vectors of a pass (NB, rounded up to 2, 4, 8) are constants.  Whole solves,
// restart 50, per Krylov iteration: 729 unknowns 87 -> 27 us, 1,584 unknowns
// 138 -> 60 us (57k of the latter's 117k cycles are the pipe's time for the
// basis).  Sums run
// over 256 virtual lanes (as cta_vsum's), in an order that does not depend on
// the CTA's shape.
constexpr int BATCH_GRAM = 64;  // doubles of T per block (BLK <= 8)
template <int NT, int KV>
struct Ortho {
  static constexpr int BLK = 8;
  static constexpr int VPL = VLANES / NT;  // virtual lanes per thread
  static constexpr int VW = VLANES / 32;   // virtual warps
  // the block in registers, or read again where it does not fit them
  static constexpr bool KEEP = VPL * KV <= 8;
  struct Vec { double x[VPL][KV]; };
  static __device__ __forceinline__ void load(Vec& v, const double* __restrict__ V, int n, bool use) {
#pragma unroll
    for (int p = 0; p < VPL; p++)
#pragma unroll
      for (int k = 0; k < KV; k++) {
        const int at = (int)threadIdx.x + p * NT + VLANES * k;
        v.x[p][k] = use && at < n ? V[at] : 0.0;
      }
  }

  // the N sums of this warp's virtual warps into part[vw][N], N a power of two
  template <int N>
  static __device__ __forceinline__ void reduce(double (&s)[VPL][N], double* part) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int p = 0; p < VPL; p++) {
      int off = 16;
#pragma unroll
      for (int m = N; m > 1; m >>= 1, off >>= 1) {  // halve the values, keep the half of the lane's bit
        const bool hi = lane & off;
#pragma unroll
        for (int l = 0; l < N / 2; l++)
          if (l < m / 2) {
            const double mine = hi ? s[p][l + m / 2] : s[p][l], give = hi ? s[p][l] : s[p][l + m / 2];
            s[p][l] = mine + __shfl_xor_sync(0xffffffffu, give, off);
          }
      }
      double t = s[p][0];
#pragma unroll
      for (; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane % (32 / N) == 0) part[(wid + p * (NT / 32)) * N + lane / (32 / N)] = t;
    }
  }
  // lane i holds sum i % N
  template <int N>
  static __device__ __forceinline__ double combine(const double* part) {
    constexpr int M = N < 4 ? 4 : N;  // (two sums are added up twice over)
    const int lane = threadIdx.x & 31, i = lane % N, g = lane / M;
    constexpr int G = 32 / M;  // groups of lanes
    double t = part[g * N + i];
#pragma unroll
    for (int k = 1; k < VW / G; k++) t += part[(g + k * G) * N + i];
#pragma unroll
    for (int off = M; off < 32; off <<= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
  }

  template <int N>
  static __device__ __forceinline__ void dot(const Vec& u, const Vec& w, int l, double (&s)[VPL][N]) {
#pragma unroll
    for (int p = 0; p < VPL; p++) {
      s[p][l] = u.x[p][0] * w.x[p][0];
#pragma unroll
      for (int k = 1; k < KV; k++) s[p][l] += u.x[p][k] * w.x[p][k];
    }
  }
  // w -= the nb <= NB vectors' parts; hc gets the coefficients, v the vectors
  template <int NB>
  static __device__ __forceinline__ void pass(const double* __restrict__ V, int n, int nb, double* hc,
                                              const double* Tm, double* part, Vec& w, Vec (&v)[KEEP ? BLK : 1]) {
    constexpr int N = NB <= 2 ? 2 : (NB <= 4 ? 4 : 8);
    const int lane = threadIdx.x & 31;
    double s[VPL][N];
    if (KEEP) {
#pragma unroll
      for (int l = 0; l < NB; l++) load(v[l], V + (int64_t)l * n, n, l < nb);
    }
#pragma unroll
    for (int l = 0; l < N; l++) {
      if (l >= NB) {
#pragma unroll
        for (int p = 0; p < VPL; p++) s[p][l] = 0.0;
        continue;
      }
      Vec& u = v[KEEP ? l : 0];
      if (!KEEP) load(u, V + (int64_t)l * n, n, l < nb);
      dot(u, w, l, s);
    }
    reduce<N>(s, part);
    __syncthreads();
    const double t = combine<N>(part);
    // h = T s: lane (i, g) takes the columns g, g + 32 / BLK, ... of row i
    const int i = lane % BLK, g = lane / BLK;
    double h = 0.0;
#pragma unroll
    for (int c = 0; c < N; c += 32 / BLK) {
      const int col = c + g;
      const double sc = __shfl_sync(0xffffffffu, t, col % N);
      if (col < N) h += Tm[i * BLK + col] * sc;
    }
    constexpr int GU = N < 32 / BLK ? N : 32 / BLK;  // groups that hold a column
    static_assert((GU & (GU - 1)) == 0, "");
#pragma unroll
    for (int off = BLK; off < BLK * GU; off <<= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
    if (threadIdx.x < nb) hc[threadIdx.x] = h;
#pragma unroll
    for (int l = 0; l < NB; l++) {
      const double hl = __shfl_sync(0xffffffffu, h, l);
      Vec& u = v[KEEP ? l : 0];
      if (!KEEP) load(u, V + (int64_t)l * n, n, l < nb);
#pragma unroll
      for (int p = 0; p < VPL; p++)
#pragma unroll
        for (int k = 0; k < KV; k++) w.x[p][k] -= hl * u.x[p][k];
    }
  }
  // the products of w with v[0..R) and, last, with itself: lane l < R holds
  // product l, every lane the square in nn
  template <int R>
  static __device__ __forceinline__ double norm(const double* __restrict__ V, int n, int r, const Vec& w,
                                                Vec (&v)[KEEP ? BLK : 1], double* part, double& nn) {
    constexpr int N = R + 1 <= 2 ? 2 : (R + 1 <= 4 ? 4 : 8);
    double s[VPL][N];
#pragma unroll
    for (int l = 0; l < N; l++) {
      if (l == N - 1) {
        dot(w, w, l, s);
      } else {  // (products beyond the block's r vectors are not read)
        Vec& u = v[KEEP ? l : 0];
        if (!KEEP) load(u, V + (int64_t)l * n, n, l < r);
        dot(u, w, l, s);
      }
    }
    reduce<N>(s, part);
    __syncthreads();
    const double t = combine<N>(part);
    nn = __shfl_sync(0xffffffffu, t, N - 1);
    return t;
  }

  // hc[0..j] = the coefficients on V[0..j] of w, whose values stand at V[j + 1]
  // (f32: in FP32); V[j + 1] <- the rest over its norm, which is returned.  tm: T of
  // every block; part: scratch.
  static __device__ __noinline__ double run(double* __restrict__ V, int n, int j, double* hc, double* tm,
                                            double* part, bool f32) {
    const int lane = threadIdx.x & 31;
    Vec w, v[KEEP ? BLK : 1];
    if (KEEP)
#pragma unroll
      for (int l = 0; l < BLK; l++) load(v[l], V, 0, false);  // zeros
    double* W = V + (int64_t)(j + 1) * n;
#pragma unroll
    for (int p = 0; p < VPL; p++)
#pragma unroll
      for (int k = 0; k < KV; k++) {
        const int at = (int)threadIdx.x + p * NT + VLANES * k;
        if (!f32) w.x[p][k] = at < n ? W[at] : 0.0;
        else w.x[p][k] = at < n ? (double)((const float*)W)[at] : 0.0;
      }
    int buf = 0, b0 = 0;
    auto scratch = [&]() {  // two in turn: a pass's barrier ends the reads of the one before
      buf ^= 1;
      return part + buf * VW * 8;
    };
    for (; b0 + BLK <= j + 1; b0 += BLK)
      pass<BLK>(V + (int64_t)b0 * n, n, BLK, hc + b0, tm + (b0 / BLK) * BATCH_GRAM, scratch(), w, v);
    const int r = j + 1 - b0;  // vectors of the last, part block: the place of the new one there
    const double* Vb = V + (int64_t)b0 * n;
    double* T0 = tm + (b0 / BLK) * BATCH_GRAM;
    if (r > 4) pass<BLK>(Vb, n, r, hc + b0, T0, scratch(), w, v);
    else if (r > 2) pass<4>(Vb, n, r, hc + b0, T0, scratch(), w, v);
    else if (r > 0) pass<2>(Vb, n, r, hc + b0, T0, scratch(), w, v);
    // the norm, and the products with the vectors of the new one's block
    double nn, t;
    if (r > 3) t = norm<BLK - 1>(Vb, n, r, w, v, scratch(), nn);
    else if (r > 1) t = norm<3>(Vb, n, r, w, v, scratch(), nn);
    else t = norm<1>(Vb, n, r, w, v, scratch(), nn);
    const bool ok = nn > 0.0 && nn < INFINITY;
    const double inv = ok ? rsqrt(nn) : 0.0;
    if (threadIdx.x < 32) {  // row r of T
      const double gl = t * inv;
      double acc = lane == r ? 1.0 : 0.0;
      for (int l = 0; l < r; l++) {
        const double g = __shfl_sync(0xffffffffu, gl, l);
        if (lane <= l) acc -= g * T0[l * BLK + lane];
      }
      if (r == 0)
        for (int e = lane; e < BLK * BLK; e += 32) T0[e] = 0.0;
      __syncwarp();
      if (lane < BLK) T0[r * BLK + lane] = acc;
    }
#pragma unroll
    for (int p = 0; p < VPL; p++)
#pragma unroll
      for (int k = 0; k < KV; k++) {
        const int at = (int)threadIdx.x + p * NT + VLANES * k;
        if (at < n) W[at] = ok ? w.x[p][k] * inv : w.x[p][k];
      }
    return ok ? nn * inv : nn;
  }
};

// by the values per virtual lane
constexpr int ORTHO_MAX = 8 * VLANES;
template <int NT>
__device__ __forceinline__ double cta_ortho(double* V, int n, int j, double* hc, double* tm, double* part, bool f32) {
  switch ((n + VLANES - 1) / VLANES) {
    case 1: return Ortho<NT, 1>::run(V, n, j, hc, tm, part, f32);
    case 2: return Ortho<NT, 2>::run(V, n, j, hc, tm, part, f32);
    case 3: return Ortho<NT, 3>::run(V, n, j, hc, tm, part, f32);
    case 4: return Ortho<NT, 4>::run(V, n, j, hc, tm, part, f32);
    case 5: return Ortho<NT, 5>::run(V, n, j, hc, tm, part, f32);
    case 6: return Ortho<NT, 6>::run(V, n, j, hc, tm, part, f32);
    case 7: return Ortho<NT, 7>::run(V, n, j, hc, tm, part, f32);
    default: return Ortho<NT, 8>::run(V, n, j, hc, tm, part, f32);
  }
}

// w against V[0..j] one vector after another, for requests whose vectors do
// not fit the registers
__device__ __forceinline__ double cta_mgs(double* V, int64_t n, int j, double* hc, double* sh8, double* slot) {
  double* w = V + (int64_t)(j + 1) * n;
  for (int i = 0; i <= j; i++) {
    const double* vi = V + (int64_t)i * n;
    const double h = cta_dot(w, vi, n, sh8, slot);
    for (int64_t k = threadIdx.x; k < n; k += blockDim.x) w[k] -= h * vi[k];
    if (threadIdx.x == 0) hc[i] = h;
    __syncthreads();
  }
  const double hn = sqrt(cta_dot(w, w, n, sh8, slot));
  const double inv = 1.0 / hn;
  if (hn > 0.0)
    for (int64_t k = threadIdx.x; k < n; k += blockDim.x) w[k] *= inv;
  return hn;
}

// Restarted GMRES, right-preconditioned by the block-Jacobi, modified
// Gram-Schmidt (FP64), Givens rotations; solves K x = b from x = 0 to
// ||b - K x|| <= max(rtol ||b||, atol) or kmaxit iterations, as fe_gmres:
// every cycle starts from the residual b - K x, and in the mixed form with a
// target below 1e-4 ||b|| that residual takes FP64 products and an estimate
// at the target sends the iterate back to it (mixed-precision iterative
// refinement).  H, the rotations and the projected right-hand side live in
// shared memory.  Returns the iterations; *res the final residual (estimate).
template <int ORDER, class T, int NT>
__device__ __noinline__ int cta_gmres(const BatchReq& q, const double* b, double* x, double rtol, double atol,
                                      double* sh, double* sh8, double* slot, double* res) {
  const int64_t n = 3 * (int64_t)q.nn;
  const int m = q.restart;
  double* H = sh;                // [(m+1) m] column j at H + j (m+1)
  double* cs = H + (m + 1) * m;  // [m]
  double* sn = cs + m;           // [m]
  double* g = sn + m;            // [m+1]
  double* y = g + m + 1;         // [m]
  double* part = y + m;          // [2][256 / 32][8]
  double* tm = part + 2 * VLANES / 32 * 8;  // [m / 8 + 1][BATCH_GRAM]
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) x[i] = 0.0;
  const double bnorm = sqrt(cta_dot(b, b, n, sh8, slot));
  const double target = fmax(rtol * bnorm, atol);
  const bool refine = sizeof(T) == 4 && target < 1e-4 * bnorm;
  double* r = q.gr;  // residual of the current iterate
  int its = 0;
  bool first = true;
  for (;;) {
    // r = b - K x (x = 0 on the first cycle)
    if (first) {
      cta_axpby(1.0, b, 0.0, r, n);
    } else {
      if (refine) cta_spmv<ORDER, T, double>(q, x, r);
      else cta_spmv<ORDER, T, T>(q, x, r);
      __syncthreads();
      for (int64_t k = threadIdx.x; k < n; k += blockDim.x) r[k] = b[k] - r[k];
    }
    __syncthreads();
    const double beta = first ? bnorm : sqrt(cta_dot(r, r, n, sh8, slot));
    first = false;
    *res = beta;
    if (beta <= target || beta == 0.0 || its >= q.kmaxit || !isfinite(beta)) break;
    double* v0 = q.V;
    cta_axpby(1.0 / beta, r, 0.0, v0, n);
    if (threadIdx.x == 0) g[0] = beta;
    if (threadIdx.x < BATCH_GRAM) tm[threadIdx.x] = threadIdx.x == 0 ? 1.0 : 0.0;  // T of the first vector's block
    __syncthreads();
    int j = 0;
    bool stop = false;
    for (; j < m && its < q.kmaxit; j++) {
      double* vj = q.V + (int64_t)j * n;
      double* w = q.V + (int64_t)(j + 1) * n;
      T* zt = (T*)q.zb;
      cta_pc<T>(q, vj, zt);
      __syncthreads();
      double* hc = H + j * (m + 1);
      double hn;
      if (n <= ORTHO_MAX) {
        cta_spmv<ORDER, T, T>(q, zt, (T*)w);
        __syncthreads();
        hn = cta_ortho<NT>(q.V, (int)n, j, hc, tm, part, sizeof(T) == 4);
      } else {
        cta_spmv<ORDER, T, T>(q, zt, w);
        __syncthreads();
        hn = cta_mgs(q.V, n, j, hc, sh8, slot);
      }
      if (threadIdx.x < 32) {  // rotations: one multiplication-addition per step in the chain, the rest across lanes
        __syncwarp();
        double a = hc[0];
        for (int i0 = 0; i0 < j; i0 += 32) {
          const int i = i0 + (int)threadIdx.x, cnt = min(32, j - i0);
          const double c = i < j ? hc[i + 1] : 0.0, ci = i < j ? cs[i] : 1.0, si = i < j ? -sn[i] : 0.0;
          const double ch = ci * c;
          double mine = 0.0;
          for (int k = 0; k < cnt; k++) {
            const double qk = __shfl_sync(0xffffffffu, ch, k), sk = __shfl_sync(0xffffffffu, si, k);
            if ((int)threadIdx.x == k) mine = a;
            a = qk + sk * a;
          }
          if (i < j) hc[i] = ci * mine - si * c;
          __syncwarp();
        }
        if (threadIdx.x == 0) {
          const double d2 = a * a + hn * hn;
          const double id = rsqrt(d2), den = d2 > 0.0 && d2 < INFINITY ? d2 * id : d2;
          cs[j] = den > 0.0 ? a * id : 1.0;
          sn[j] = den > 0.0 ? hn * id : 0.0;
          hc[j] = den;
          hc[j + 1] = 0.0;
          g[j + 1] = -sn[j] * g[j];
          g[j] = cs[j] * g[j];
        }
      }
      __syncthreads();
      its++;
      if (fabs(g[j + 1]) <= target || hn == 0.0) {
        stop = hn == 0.0;
        j++;
        break;
      }
    }
    const int kdim = j;
    const double est = fabs(g[kdim]);
    if (threadIdx.x < 32) {  // back substitution H y = g, a column at a time (g is spent)
      for (int i = kdim - 1; i >= 0; i--) {
        const double yi = g[i] / H[i * (m + 1) + i];
        __syncwarp();
        for (int l = threadIdx.x; l < i; l += 32) g[l] -= H[i * (m + 1) + l] * yi;
        if (threadIdx.x == 0) y[i] = yi;
        __syncwarp();
      }
    }
    __syncthreads();
    // x += D^{-1} (V y)
    double* u = q.zb;
    for (int64_t k = threadIdx.x; k < n; k += blockDim.x) {
      double s = 0.0;
      for (int i = 0; i < kdim; i++) s += y[i] * q.V[(int64_t)i * n + k];
      u[k] = s;
    }
    __syncthreads();
    double* pu = q.V;  // the basis is spent: preconditioned correction
    cta_pc<T>(q, (const double*)u, pu);
    __syncthreads();
    for (int64_t k = threadIdx.x; k < n; k += blockDim.x) x[k] += pu[k];
    __syncthreads();
    *res = est;
    // the estimate decides, except in the refined mixed form, where an
    // estimate at the target goes back to the top for the FP64-product residual
    if (its >= q.kmaxit || stop || !isfinite(est) || (est <= target && !refine)) break;
  }
  return its;
}

template <int ORDER, class T>
__device__ void cta_record(const BatchReq& q, int k, double rk, int lit, double eta) {
  if (threadIdx.x == 0 && k < BATCH_HIST) {
    q.out->res_hist[k] = rk;
    q.out->lit_hist[k] = lit;
    q.out->eta_hist[k] = eta;
    q.out->hist_len = k + 1;
  }
}

template <int ORDER, class T, int NT>
__global__ void __launch_bounds__(NT) k_batch_solve(const BatchReq* __restrict__ reqs) {
  __shared__ BatchReq q;
  __shared__ double slot;
  __shared__ double sh8[VLANES / 32];
  extern __shared__ __align__(16) unsigned char smraw[];
  if (threadIdx.x == 0) q = reqs[blockIdx.x];
  __syncthreads();
  // GMRES scratch after the tangent's staging area
  double* sh = (double*)(smraw + ((sizeof(T) * TanCfg<ORDER, T>::EPB * TanCfg<ORDER, T>::PER_E + 15) / 16) * 16);
  const int64_t n = 3 * (int64_t)q.nn;
  double* d = q.d;
  double rk = cta_residual<ORDER>(q, d, q.r, sh8, &slot);
  const double r0 = rk;
  int status = NL_MAX_IT, nit = 0, assemblies = 0;
  int64_t lit_total = 0;
  cta_record<ORDER, T>(q, 0, r0, 0, 0.0);
  if (!isfinite(r0)) status = NL_NONFINITE;
  else if (r0 == 0.0) status = FE_OK;
  else if (q.method == NL_NK || q.method == NL_INK) {
    double eta = q.method == NL_NK ? q.ksp_rtol : q.ew0;
    const double alpha2 = 0.5 * (1.0 + sqrt(5.0));
    for (int k = 1; k <= q.max_it; k++) {
      cta_tangent<ORDER, T>(q, d);
      assemblies++;
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) q.t[i] = -q.r[i];
      __syncthreads();
      double lres_est = 0.0;
      const int its = cta_gmres<ORDER, T, NT>(q, q.t, q.dl, eta, q.ksp_atol, sh, sh8, &slot, &lres_est);
      lit_total += its;
      // linear residual ||R + K delta|| with FP64 products (Eisenstat-Walker)
      cta_spmv<ORDER, T, double>(q, (const double*)q.dl, q.rn);
      __syncthreads();
      const double* rr = q.r;
      const double* rl = q.rn;
      const double lnorm = sqrt(cta_vsum(
          n, [&](int64_t i) { const double v = rl[i] + rr[i]; return v * v; }, sh8, &slot));
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) d[i] += q.dl[i];
      __syncthreads();
      const double rprev = rk;
      rk = cta_residual<ORDER>(q, d, q.r, sh8, &slot);
      nit = k;
      cta_record<ORDER, T>(q, k, rk, its, eta);
      if (!isfinite(rk)) { status = NL_NONFINITE; break; }
      if (rk <= q.tol * r0) { status = FE_OK; break; }
      if (rk > q.dtol * r0) { status = NL_DIVERGED; break; }
      if (q.method == NL_INK) {
        const double eta_prev = eta;
        eta = fabs(rk - lnorm) / rprev;
        const double stol = pow(eta_prev, alpha2);
        if (stol > 0.1) eta = fmax(eta, stol);
        eta = fmin(eta, q.ewmax);
      }
    }
  } else {  // B / iB
    cta_tangent<ORDER, T>(q, d);
    assemblies = 1;
    __shared__ double alpha[BATCH_HIST];
    __shared__ double rho[BATCH_HIST];
    int head = 0, np = 0;
    const int mcap = min(q.mcap, BATCH_HIST);
    for (int k = 1; k <= q.max_it; k++) {
      // two-loop: z = H R, newest pair first
      double* z = q.t;
      cta_axpby(1.0, q.r, 0.0, q.w, n);  // q-vector of the recursion
      __syncthreads();
      for (int l = np - 1; l >= 0; l--) {
        const int sl = (head + l) % mcap;
        const double* s = q.S + (int64_t)sl * n;
        const double* yv = q.Y + (int64_t)sl * n;
        const double a = rho[sl] * cta_dot(s, q.w, n, sh8, &slot);
        if (threadIdx.x == 0) alpha[sl] = a;
        cta_axpby(-a, yv, 1.0, q.w, n);
        __syncthreads();
      }
      int its = 0;
      if (q.method == NL_B) {
        cta_pc<T>(q, (const double*)q.w, z);
      } else {
        double est = 0.0;
        its = cta_gmres<ORDER, T, NT>(q, q.w, z, q.ksp_rtol, q.ksp_atol, sh, sh8, &slot, &est);
      }
      __syncthreads();
      lit_total += its;
      for (int l = 0; l < np; l++) {
        const int sl = (head + l) % mcap;
        const double* s = q.S + (int64_t)sl * n;
        const double* yv = q.Y + (int64_t)sl * n;
        const double bcoef = rho[sl] * cta_dot(yv, z, n, sh8, &slot);
        cta_axpby(alpha[sl] - bcoef, s, 1.0, z, n);
        __syncthreads();
      }
      // delta = -z; d += delta; new residual; secant pair
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        q.dl[i] = -z[i];
        d[i] -= z[i];
      }
      __syncthreads();
      rk = cta_residual<ORDER>(q, d, q.rn, sh8, &slot);
      nit = k;
      cta_record<ORDER, T>(q, k, rk, its, q.method == NL_B ? 0.0 : q.ksp_rtol);
      const double* rr = q.r;
      const double* rl = q.rn;
      const double* dd = q.dl;
      const double ys = cta_vsum(n, [&](int64_t i) { return (rl[i] - rr[i]) * dd[i]; }, sh8, &slot);
      if (ys > 0.0) {
        const int sl = np < mcap ? (head + np) % mcap : head;
        double* s = q.S + (int64_t)sl * n;
        double* yv = q.Y + (int64_t)sl * n;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
          s[i] = q.dl[i];
          yv[i] = q.rn[i] - q.r[i];
        }
        if (threadIdx.x == 0) rho[sl] = 1.0 / ys;
        if (np < mcap) np++;
        else head = (head + 1) % mcap;
      }
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) q.r[i] = q.rn[i];
      __syncthreads();
      if (!isfinite(rk)) { status = NL_NONFINITE; break; }
      if (rk <= q.tol * r0) { status = FE_OK; break; }
      if (rk > q.dtol * r0) { status = NL_DIVERGED; break; }
      status = NL_MAX_IT;
    }
  }
  if (threadIdx.x == 0) {
    fe_batch_out* o = q.out;
    o->status = status;
    o->nit = nit;
    o->lit_total = lit_total;
    o->assemblies = assemblies;
    o->r0 = r0;
    o->rfinal = rk;
  }
}

// the kernels of one order, each order in a translation unit of its own (the
// orthogonalisation is instantiated per kernel: together they took twice as
// long to compile as the rest of the library)
template <int ORDER>
const void* batch_kernel(bool f64, int nt) {
  if (f64) return nt == 128 ? (const void*)k_batch_solve<ORDER, double, 128> : (const void*)k_batch_solve<ORDER, double, 256>;
  return nt == 128 ? (const void*)k_batch_solve<ORDER, float, 128> : (const void*)k_batch_solve<ORDER, float, 256>;
}
const void* fe_batch_kernel_p1(bool f64, int nt);
const void* fe_batch_kernel_p2(bool f64, int nt);
