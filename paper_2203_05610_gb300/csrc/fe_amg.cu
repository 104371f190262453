// fe_amg.cu -- smoothed-aggregation algebraic multigrid (AMG) on the nodal
// blocks, as the preconditioner of the displacement block.
//
// The paper preconditions its Krylov solves with algebraic multigrid on
// blocks of size 3 (BoomerAMG with bs = 3, Section "Test problems and
// solvers details" and Appendix A) without describing it; this is a
// smoothed-aggregation V-cycle of that class:
//   - aggregation on the block graph of A_l (nodes whose components are all
//     absent -- Dirichlet at level 0 -- left out, no strength filter): roots
//     = greedy maximal distance-2 independent set in descending
//     splitmix64(node) priority, ties by id; a root takes its neighbours;
//     every other node joins the aggregate of its smallest-id neighbour
//     taken so; aggregates numbered by root id;
//   - near null space: the six rigid motions (translations, rotations
//     (-y, x, 0), (0, -z, y), (z, 0, -x)); tentative prolongator T by
//     modified Gram-Schmidt QR of each aggregate's rows (columns left with
//     <= 1e-8 of their norm are dropped and that coarse component is
//     absent); coarse nodes carry 6 components;
//   - P = (I - omega D^-1 A) T, omega = 4 / (3 rho), rho from 15 power steps
//     on D^-1 A (D the block diagonal) from x_k = u(splitmix64(k)) - 1/2;
//   - Galerkin A_{l+1} = P^T A_l P, absent components with a unit diagonal;
//   - Chebyshev smoothing of degree 2 in D^-1 A on [rho/30, 1.1 rho] before
//     and after the coarse correction; exact solve on the coarsest level
//     (<= 16 nodes) with the inverse from Gauss-Jordan elimination.
//
// GB300 design.  Everything that depends only on the mesh -- the
// aggregates, T (rigid motions at the node coordinates), the patterns of P,
// A P, P^T and every coarse operator, and the index lists of the Galerkin
// products -- is built once per mesh on the host (native C++, like the
// mesh's own block pattern) and kept resident.  What depends on the
// tangent's values runs on the device after every assembly: block
// inverses, power iterations, P, A P, P^T A P and the coarsest inverse,
// each output entry computed by one thread from a fixed gather list (no
// atomics: deterministic, and the same summation order as a plain loop).
// The numbers are formed in FP64 for an FP64 tangent and in FP32 for the
// mixed forms (GB300's FP32 rate is tens of times its FP64 rate); the
// V-cycle runs in the tangent's precision (FP32 values, vectors and
// accumulation in the mixed forms), the coarsest inverse is formed in FP64.  A
// Chebyshev step is one fused kernel: the SpMV with A_l, the residual update,
// the block-Jacobi product and the direction and iterate updates of its
// rows (r stays b - A x throughout, so the residual for the restriction
// comes for free); level 0 reads the tangent in its tiled layout, coarser
// levels their 6x6 blocks block-major with 16-byte loads.  FP32 levels of at
// most VC_BOTTOM_MAXNNZ blocks below level 0 run in one thread block (one launch
// instead of seven or more latency-bound ones), and the whole V-cycle is
// captured as one CUDA graph.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <numeric>
#include <type_traits>
#include <vector>

#include "fe_internal.h"
#include "fe_stream.cuh"

namespace {

constexpr int AMG_MAXLEV = 12;
constexpr int AMG_COARSE = 16;   // the coarsest level has at most this many nodes
constexpr int AMG_NS = 6;        // near null space vectors
constexpr int AMG_DENSE_MAX = 96;
constexpr int AMG_POWER_STEPS = 15;
constexpr double AMG_QR_DROP = 1e-8;
// one level's device scalars (AmgHier::scal): spectral radius, last sum of
// squares, next scale factor, prolongator weight
constexpr int SC_RHO = 0, SC_SS = 1, SC_F = 2, SC_OMEGA = 3, SC_N = 4;

uint64_t mix64(uint64_t z) {  // splitmix64 (Steele, Lea and Flood; Vigna's constants)
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t mix64_d(uint64_t z) {
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

}  // namespace

struct AmgLevel {
  int n = 0, b = 3, nc = 0;
  int64_t nnz = 0, nnzp = 0, nnzap = 0, nnzr = 0, napidx = 0, nralist = 0;
  // structure (device)
  const int* ptr = nullptr;  // A_l pattern (level 0: the mesh's)
  const int* col = nullptr;
  const int* diag = nullptr; // [n] diagonal block positions
  int* own = nullptr;        // one allocation holding this level's int arrays
  unsigned char* absent = nullptr;
  int *agg = nullptr, *pptr = nullptr, *pcol = nullptr, *prow = nullptr;
  int2* pk_ptr = nullptr;    // the blocks of each P entry (k_amg_plists), its place in R
  int *pk = nullptr, *rpos = nullptr;
  int64_t *apoff = nullptr, *raoff = nullptr;  // starts of each fine row's places, each coarse row's products below
  // places of the products in their A P row (k_amg_ap), and (P entry, A P
  // entry) of the products of each entry of A_{l+1} (k_amg_rap); optional, null
  // where they do not fit (fe_amg_release_lists)
  int* apidx = nullptr;
  int2* ralist = nullptr;
  int64_t* lend = nullptr;                // their ends
  int* crow = nullptr;                    // row of each entry of A_{l+1}
  float* tnode32 = nullptr;               // tnode in FP32
  int *rptr = nullptr, *rcol = nullptr, *rsrc = nullptr;
  int *apptr = nullptr, *apcol = nullptr;
  double* tnode = nullptr;   // [n][b*6] tentative block of each node
  // numbers (device)
  double* val64 = nullptr;  // level >= 1: [nnz][b*b]
  float* val32 = nullptr;
  double* dinv64 = nullptr;
  float* dinv32 = nullptr;
  double *p64 = nullptr, *r64 = nullptr, *ap64 = nullptr;
  float *p32 = nullptr, *r32 = nullptr, *ap32 = nullptr;
  double* inv64 = nullptr;
  float* inv32 = nullptr;
  double rho = 0.0;
  double* pt64 = nullptr;    // tiled V-cycle copy of P_l
  float* pt32 = nullptr;
  double* coef64 = nullptr;  // Chebyshev coefficients {1/theta, c1, c2} in device memory, so
  float* coef32 = nullptr;   // a captured V-cycle stays valid when a new tangent changes them
  // V-cycle vectors [n*b] in the V-cycle precision (level 0: x is the mesh's
  // SpMV input zx)
  void *x = nullptr, *r = nullptr, *d0 = nullptr, *d1 = nullptr, *e = nullptr;
};

struct AmgHier {
  int nlev = 0;
  AmgLevel lev[AMG_MAXLEV];
  int vec_elem = 0;          // bytes per V-cycle vector element allocated (0: none yet)
  double* pw = nullptr;      // power iterations: x, y [2][max n*b]
  double* part = nullptr;    // partial sums of a power step, one per block
  unsigned* ticket = nullptr;
  double* scal = nullptr;    // [AMG_MAXLEV][SC_N]
  std::vector<void*> allocs; // device buffers owned by the hierarchy
  int64_t bytes = 0;         // their size (counted in the mesh's device bytes)
  bool ready = false;        // numbers formed for the current tangent
  int prec = -1;             // its precision
  // the V-cycle captured as a CUDA graph, output lev[0].x; its first kernel
  // reads the caller's vector (argument `root_arg` of node `root`, set before
  // each launch)
  cudaGraph_t graph = nullptr;
  cudaGraphNode_t root = nullptr;
  int root_arg = 0;
  StreamShape shape0{};             // the streamed level-0 step's launch and row ranges
  int* part0 = nullptr;             // [shape0.ranges + 1]
  int part0_len = 0;
  cudaStream_t cap = nullptr;       // capture stream (the mesh's may be the legacy stream)
  cudaGraphExec_t exec = nullptr;
  int exec_prec = -1;               // tangent precision the graph was captured for
  double vc_bytes = 0, vc_flops = 0; // algorithmic bytes and flops of one V-cycle
};

namespace {

// ---------------------------------------------------------------- host structure
struct HostLevel {
  int n = 0, b = 3, nc = 0;
  std::vector<int> ptr, col, diag;
  std::vector<uint8_t> absent;
  std::vector<double> ns;  // [n*b][6]
  std::vector<int> agg, pptr, pcol, rptr, rcol, rsrc, apptr, apcol;
  std::vector<double> tnode;  // [n][b*6]
  std::vector<int64_t> apoff, raoff;
};

uint8_t full_mask(int b) { return (uint8_t)((1u << b) - 1u); }

// sorted unique values of v[beg, end) appended to out; returns the new size
void sort_unique(std::vector<int>& tmp) {
  std::sort(tmp.begin(), tmp.end());
  tmp.erase(std::unique(tmp.begin(), tmp.end()), tmp.end());
}

void aggregate(HostLevel& L) {
  const int n = L.n;
  const uint8_t full = full_mask(L.b);
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::vector<uint64_t> pri(n);
  for (int i = 0; i < n; i++) pri[i] = mix64((uint64_t)i);
  std::sort(order.begin(), order.end(), [&](int a, int c) { return pri[a] != pri[c] ? pri[a] > pri[c] : a < c; });
  std::vector<int> root(n, -1);  // root whose neighbourhood took the node
  for (int i : order) {
    if (L.absent[i] == full || root[i] >= 0) continue;
    bool taken = false;
    for (int k = L.ptr[i]; k < L.ptr[i + 1] && !taken; k++) {
      const int j = L.col[k];
      taken = j != i && L.absent[j] != full && root[j] >= 0;
    }
    if (taken) continue;
    for (int k = L.ptr[i]; k < L.ptr[i + 1]; k++)
      if (L.absent[L.col[k]] != full) root[L.col[k]] = i;
    root[i] = i;
  }
  std::vector<int> id(n, -1);
  L.nc = 0;
  for (int i = 0; i < n; i++)
    if (root[i] == i) id[i] = L.nc++;
  L.agg.assign(n, -1);
  for (int i = 0; i < n; i++)
    if (root[i] >= 0) L.agg[i] = id[root[i]];
  for (int i = 0; i < n; i++) {  // nodes at distance 2 from every root
    if (L.absent[i] == full || root[i] >= 0) continue;
    for (int k = L.ptr[i]; k < L.ptr[i + 1]; k++) {
      const int j = L.col[k];
      if (j != i && root[j] >= 0) {
        L.agg[i] = id[root[j]];
        break;
      }
    }
  }
}

// T per node, coarse near null space and absent components, all patterns
// of the level's products and the coarse level's pattern
void coarsen(HostLevel& L, HostLevel& C) {
  const int n = L.n, nc = L.nc, b = L.b, K = AMG_NS;
  std::vector<std::vector<int>> members(nc);
  for (int i = 0; i < n; i++)
    if (L.agg[i] >= 0) members[L.agg[i]].push_back(i);
  C.n = nc;
  C.b = K;
  C.absent.assign(nc, 0);
  C.ns.assign((size_t)nc * K * K, 0.0);
  L.tnode.assign((size_t)n * b * K, 0.0);
  std::vector<double> Q;
  for (int a = 0; a < nc; a++) {
    const std::vector<int>& mem = members[a];
    const int rows = (int)mem.size() * b;
    Q.assign((size_t)rows * K, 0.0);  // column c at Q[c * rows ...]
    for (size_t s = 0; s < mem.size(); s++)
      for (int i = 0; i < b; i++)
        for (int c = 0; c < K; c++) Q[(size_t)c * rows + s * b + i] = L.ns[((size_t)mem[s] * b + i) * K + c];
    double* R = C.ns.data() + (size_t)a * K * K;  // R(p, c) at R[p K + c]
    for (int c = 0; c < K; c++) {
      double* v = Q.data() + (size_t)c * rows;
      double n0 = 0.0;
      for (int t = 0; t < rows; t++) n0 += v[t] * v[t];
      n0 = std::sqrt(n0);
      for (int p = 0; p < c; p++) {
        const double* q = Q.data() + (size_t)p * rows;
        double h = 0.0;
        for (int t = 0; t < rows; t++) h += q[t] * v[t];
        R[p * K + c] = h;
        for (int t = 0; t < rows; t++) v[t] -= h * q[t];
      }
      double nv = 0.0;
      for (int t = 0; t < rows; t++) nv += v[t] * v[t];
      nv = std::sqrt(nv);
      if (n0 == 0.0 || nv <= AMG_QR_DROP * n0) {
        std::fill(v, v + rows, 0.0);
        R[c * K + c] = 0.0;
        C.absent[a] |= (uint8_t)(1u << c);
      } else {
        for (int t = 0; t < rows; t++) v[t] /= nv;
        R[c * K + c] = nv;
      }
    }
    for (size_t s = 0; s < mem.size(); s++)
      for (int i = 0; i < b; i++)
        for (int c = 0; c < K; c++) L.tnode[((size_t)mem[s] * b + i) * K + c] = Q[(size_t)c * rows + s * b + i];
  }
  const uint8_t full = full_mask(b);
  std::vector<int> tmp;
  // P: row i takes the aggregates of its neighbours
  L.pptr.assign(n + 1, 0);
  L.pcol.clear();
  for (int i = 0; i < n; i++) {
    tmp.clear();
    if (L.absent[i] != full)
      for (int k = L.ptr[i]; k < L.ptr[i + 1]; k++)
        if (L.agg[L.col[k]] >= 0) tmp.push_back(L.agg[L.col[k]]);
    sort_unique(tmp);
    L.pcol.insert(L.pcol.end(), tmp.begin(), tmp.end());
    L.pptr[i + 1] = (int)L.pcol.size();
  }
  // A P: row i takes the P rows of its neighbours
  L.apptr.assign(n + 1, 0);
  L.apcol.clear();
  L.apoff.assign(n + 1, 0);
  for (int i = 0; i < n; i++) {
    tmp.clear();
    for (int k = L.ptr[i]; k < L.ptr[i + 1]; k++) {
      const int j = L.col[k];
      tmp.insert(tmp.end(), L.pcol.begin() + L.pptr[j], L.pcol.begin() + L.pptr[j + 1]);
    }
    L.apoff[i + 1] = L.apoff[i] + (int64_t)tmp.size();
    sort_unique(tmp);
    L.apcol.insert(L.apcol.end(), tmp.begin(), tmp.end());
    L.apptr[i + 1] = (int)L.apcol.size();
  }
  // P^T: row a lists (fine node, P entry) by ascending fine node
  L.rptr.assign(nc + 1, 0);
  for (int q = 0; q < L.pptr[n]; q++) L.rptr[L.pcol[q] + 1]++;
  for (int a = 0; a < nc; a++) L.rptr[a + 1] += L.rptr[a];
  L.rcol.assign(L.pptr[n], 0);
  L.rsrc.assign(L.pptr[n], 0);
  {
    std::vector<int> fill(L.rptr.begin(), L.rptr.end() - 1);
    for (int i = 0; i < n; i++)
      for (int q = L.pptr[i]; q < L.pptr[i + 1]; q++) {
        const int s = fill[L.pcol[q]]++;
        L.rcol[s] = i;
        L.rsrc[s] = q;
      }
  }
  L.raoff.assign(nc + 1, 0);
  for (int a = 0; a < nc; a++) {
    L.raoff[a + 1] = L.raoff[a];
    for (int q = L.rptr[a]; q < L.rptr[a + 1]; q++) L.raoff[a + 1] += L.apptr[L.rcol[q] + 1] - L.apptr[L.rcol[q]];
  }
  // coarse pattern: row a takes the A P rows of its P^T row, and the diagonal
  C.ptr.assign(nc + 1, 0);
  C.col.clear();
  for (int a = 0; a < nc; a++) {
    tmp.clear();
    tmp.push_back(a);
    for (int s = L.rptr[a]; s < L.rptr[a + 1]; s++) {
      const int i = L.rcol[s];
      tmp.insert(tmp.end(), L.apcol.begin() + L.apptr[i], L.apcol.begin() + L.apptr[i + 1]);
    }
    sort_unique(tmp);
    C.col.insert(C.col.end(), tmp.begin(), tmp.end());
    C.ptr[a + 1] = (int)C.col.size();
  }
  C.diag.assign(nc, -1);
  for (int a = 0; a < nc; a++)
    for (int k = C.ptr[a]; k < C.ptr[a + 1]; k++)
      if (C.col[k] == a) C.diag[a] = k;
}

// ---------------------------------------------------------------- device helpers
// V-cycle copies of the operators are tiled like the tangent: tiles of 32
// consecutive blocks, component-major inside a tile, so the lanes of a warp
// reading one component of consecutive blocks read one 128-byte run
template <int NV>
__host__ __device__ __forceinline__ int64_t tix(int64_t k, int c) {
  return (k >> 5) * (NV * 32) + 32 * c + (k & 31);
}
inline int64_t tiled_count(int64_t nblocks, int nv) { return (nblocks + 31) / 32 * 32 * nv; }

// a stored value in the V-cycle's arithmetic type T (FP32 values stay FP32)
template <class T, class V>
__device__ __forceinline__ T ldt(const V* p) {
  if constexpr (std::is_same<V, __nv_bfloat16>::value) return (T)__bfloat162float(*p);
  else return (T)__ldg(p);
}

// a block-major 6x6 block with 16-byte loads (from a device allocation, so
// 16-byte aligned)
template <class T>
__device__ __forceinline__ void load_block6(const T* val, int64_t k, T (&v)[AMG_NS * AMG_NS]) {
  constexpr int N = AMG_NS * AMG_NS;
  if constexpr (sizeof(T) == 4) {
    const float4* p4 = reinterpret_cast<const float4*>(val + k * N);
#pragma unroll
    for (int t = 0; t < N / 4; t++) {
      const float4 u = __ldg(p4 + t);
      v[4 * t] = u.x;
      v[4 * t + 1] = u.y;
      v[4 * t + 2] = u.z;
      v[4 * t + 3] = u.w;
    }
  } else {
    const double2* p2 = reinterpret_cast<const double2*>(val + k * N);
#pragma unroll
    for (int t = 0; t < N / 2; t++) {
      const double2 u = __ldg(p2 + t);
      v[2 * t] = u.x;
      v[2 * t + 1] = u.y;
    }
  }
}

// entry c of block k, or the whole block, in the setup's arithmetic type C:
// level 0 (B = 3) reads the tangent in its tiled layout, coarser levels (B =
// 6) their block-major values
template <class C, class V, int B>
struct Vals {
  const V* v;
  __device__ __forceinline__ C operator()(int64_t k, int c) const {
    return B == 3 ? ldt<C, V>(v + kv_index(k, c)) : ldt<C, V>(v + k * (B * B) + c);
  }
  __device__ __forceinline__ void block(int64_t k, C (&a)[B * B]) const {
    if constexpr (B == 3) {
#pragma unroll
      for (int c = 0; c < 9; c++) a[c] = ldt<C, V>(v + kv_index(k, c));
    } else {
      load_block6<C>(v, k, a);
    }
  }
};

// ---------------------------------------------------------------- numeric setup kernels
// C is the setup's arithmetic type: FP64 for an FP64 tangent, FP32 for the
// mixed forms (whose V-cycle runs in FP32; GB300's FP32 rate is tens of
// times its FP64 rate).  The block inverses and the dense coarsest inverse are
// always formed in FP64, with one reciprocal per pivot (an FP64 division is
// about 7 multiplications' issue time).
template <class T>
__device__ __forceinline__ void swap_if(bool s, T& a, T& b) {
  const T t = a;
  a = s ? b : a;
  b = s ? t : b;
}

// level 0: one thread per 3x3 block, Gauss-Jordan in registers (fixed loops:
// with run-time pivot indices the matrices lived in local memory, 82 us for
// 160k blocks)
template <class C, class V>
__global__ void k_amg_dinv3(int n, const int* __restrict__ diag, Vals<C, V, 3> A, C* __restrict__ dinv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double a[3][3], v[3][3];
  const int64_t k = diag[i];  // (-1: a row without blocks, identity)
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      a[r][c] = k >= 0 ? (double)A(k, 3 * r + c) : (r == c ? 1.0 : 0.0);
      v[r][c] = r == c ? 1.0 : 0.0;
    }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    int p = c;
    double best = fabs(a[c][c]);
#pragma unroll
    for (int r = c + 1; r < 3; r++)
      if (fabs(a[r][c]) > best) {
        best = fabs(a[r][c]);
        p = r;
      }
#pragma unroll
    for (int r = c + 1; r < 3; r++)
#pragma unroll
      for (int j = 0; j < 3; j++) {
        swap_if(p == r, a[c][j], a[r][j]);
        swap_if(p == r, v[c][j], v[r][j]);
      }
    const double inv = 1.0 / a[c][c];
#pragma unroll
    for (int j = 0; j < 3; j++) {
      if (j > c) a[c][j] *= inv;
      v[c][j] *= inv;
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      if (r == c) continue;
      const double f = a[r][c];
#pragma unroll
      for (int j = 0; j < 3; j++) {
        if (j > c) a[r][j] -= f * a[c][j];
        v[r][j] -= f * v[c][j];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int c = 0; c < 3; c++) dinv[(int64_t)i * 9 + 3 * r + c] = (C)v[r][c];
}

// coarse levels: 16 lanes per 6x6 block, lane j < 12 holds column j of
// [A | I]; the pivot column's entries reach the other lanes by shuffles
template <class C, class V>
__global__ void __launch_bounds__(128) k_amg_dinv6(int n, const int* __restrict__ diag, Vals<C, V, AMG_NS> A,
                                                   C* __restrict__ dinv) {
  constexpr int B = AMG_NS;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = min(t / 16, n - 1), j = t % 16;  // (the last blocks' spare lanes repeat block n - 1)
  const int64_t k = diag[i];
  double a[B];
#pragma unroll
  for (int r = 0; r < B; r++) a[r] = j < B ? (double)A(k, B * r + j) : (j - B == r ? 1.0 : 0.0);
#pragma unroll
  for (int c = 0; c < B; c++) {
    // pivot row of column c (the first of the largest), found by lane c
    int p = c;
    double best = fabs(a[c]);
#pragma unroll
    for (int r = c + 1; r < B; r++)
      if (fabs(a[r]) > best) {
        best = fabs(a[r]);
        p = r;
      }
    p = __shfl_sync(0xffffffffu, p, c, 16);
#pragma unroll
    for (int r = c + 1; r < B; r++) swap_if(p == r, a[c], a[r]);
    double f[B];
#pragma unroll
    for (int r = 0; r < B; r++) f[r] = __shfl_sync(0xffffffffu, a[r], c, 16);
    a[c] *= 1.0 / f[c];
#pragma unroll
    for (int r = 0; r < B; r++)
      if (r != c) a[r] -= f[r] * a[c];
  }
  if (t / 16 < n && j >= B && j < 2 * B)
#pragma unroll
    for (int r = 0; r < B; r++) dinv[(int64_t)i * B * B + B * r + (j - B)] = (C)a[r];
}

template <class C>
__global__ void k_amg_start(int64_t N, C* __restrict__ x, double* __restrict__ scal) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < N) x[k] = (C)((double)(mix64_d((uint64_t)k) >> 11) * (1.0 / 9007199254740992.0) - 0.5);
  if (k == 0) {
    scal[SC_F] = 1.0;
    scal[SC_SS] = 1.0;
  }
}

// Power iteration on D^-1 A, rho = |y| / |x| of the last step.  A step is one
// kernel: the product, D^-1, the sums of squares (FP64, one partial per block)
// and, in the last block to finish, the sum of the partials in block order and
// the next factor; the last step also leaves rho, the prolongator's omega and
// the Chebyshev coefficients in device memory, so the host reads all levels'
// radii once, after the whole setup.  (Before: three kernels per step, the
// scaling one adding 512 partials in one thread of every block: 31-80 us.)
//   FP64: x_{k+1} = f_k D^-1 A x_k, f_k the power of two that brings |x_{k+1}|
// near 1 (scaling by it is exact).
//   FP32: x is y / |y| rounded to FP32, formed where it is read.  The rounding
// of the coarse operators is amplified by their condition (1e-4 to 1e-3 in a
// V-cycle's result), and one unit in the last place of omega changes all of
// it, so each FP32 sum of the setup keeps a fixed order of its own -- a row's
// blocks over 32 lanes, a product's terms in list order -- that no launch
// shape changes.
struct PowerArgs {
  double* part;      // [2][blocks]
  unsigned* ticket;
  double* scal;      // this level's SC_* values
  double* coef64;    // Chebyshev coefficients {1/theta, c1, c2}
  float* coef32;
};

// what the next step multiplies the iterate by
template <class C>
struct PowerScale;
template <>
struct PowerScale<double> {  // (applied when y was written)
  __device__ __forceinline__ explicit PowerScale(double) {}
  __device__ __forceinline__ double operator()(double y) const { return y; }
};
template <>
struct PowerScale<float> {  // y f rounded once: f = h + l, y h + its error + y l
  float h, l;
  __device__ __forceinline__ explicit PowerScale(double f) : h((float)f), l((float)(f - (double)h)) {}
  __device__ __forceinline__ float operator()(float y) const {
    const float p = y * h;
    return p + fmaf(y, l, fmaf(y, h, -p));
  }
};

// from the sums of squares ss of y and (FP32, last step) xx of x
template <class C>
__device__ __forceinline__ void power_result(const PowerArgs& a, double ss, double xx, bool last_step) {
  double rho = 0.0;
  if (sizeof(C) == 8) {
    const double f = a.scal[SC_F];
    rho = sqrt(ss) / (sqrt(a.scal[SC_SS]) * f);
    a.scal[SC_SS] = ss;
    a.scal[SC_F] = ss > 0.0 && isfinite(ss) ? ldexp(1.0, -(ilogb(ss) >> 1)) : 1.0;
  } else {
    a.scal[SC_F] = 1.0 / sqrt(ss);
    if (last_step) rho = sqrt(ss) / sqrt(xx);
  }
  if (!last_step) return;
  a.scal[SC_RHO] = rho;
  a.scal[SC_OMEGA] = 4.0 / (3.0 * rho);
  const double lo = rho / 30.0, hi = 1.1 * rho;
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
  const double r0 = 1.0 / sigma, r1 = 1.0 / (2.0 * sigma - r0);
  const double c[3] = {1.0 / theta, r1 * r0, 2.0 * r1 / delta};
  for (int q = 0; q < 3; q++) {
    a.coef64[q] = c[q];
    a.coef32[q] = (float)c[q];
  }
}

// block sum of ss (result in thread 0); every thread of the block calls it
__device__ __forceinline__ double power_block_sum(double ss, double* sh) {
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = ss;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = (int)threadIdx.x < (int)(blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

template <class C>
__device__ __forceinline__ void power_finish(const PowerArgs& a, double ss, double xx, double* sh, bool last_step) {
  __shared__ bool last;
  const bool two = sizeof(C) == 4 && last_step;
  const double bs = power_block_sum(ss, sh), bx = two ? power_block_sum(xx, sh) : 0.0;
  if (threadIdx.x == 0) {
    a.part[blockIdx.x] = bs;
    if (two) a.part[gridDim.x + blockIdx.x] = bx;
    __threadfence();
    last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0, t = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    s += ((volatile double*)a.part)[b];
    if (two) t += ((volatile double*)a.part)[gridDim.x + b];
  }
  s = power_block_sum(s, sh);
  if (two) t = power_block_sum(t, sh);
  if (threadIdx.x == 0) {
    *a.ticket = 0u;
    power_result<C>(a, s, t, last_step);
  }
}

template <class C>
struct EpiPower {
  const C* dinv;
  C* y;
  C f;
  double ss;
  C di[9];
  __device__ __forceinline__ void prefetch(int, int, int) {}
  __device__ __forceinline__ void load(int r0, int, int nd, int lane) {
    if (lane < nd)
#pragma unroll
      for (int q = 0; q < 9; q++) di[q] = dinv[9 * (int64_t)(r0 + lane) + q];
  }
  __device__ __forceinline__ void finish(int row, const C (&s)[3]) {
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const C v = f * (di[3 * q] * s[0] + di[3 * q + 1] * s[1] + di[3 * q + 2] * s[2]);
      y[3 * (int64_t)row + q] = v;
      ss += (double)v * (double)v;
    }
  }
};

// level 0 in FP64: the streamed product of fe_stream.cuh
template <class C, class V>
__global__ void __launch_bounds__(STREAM_THREADS, stream_blocks_per_sm<C>())
    k_amg_power0(int n, int warps, int ranges, const int* __restrict__ part, const int* __restrict__ row_ptr,
                 const int* __restrict__ col, const V* __restrict__ val, const C* __restrict__ dinv,
                 const C* __restrict__ x, C* __restrict__ y, PowerArgs a, bool last_step) {
  __shared__ StreamShared<C> sh;
  __shared__ double red[32];
  const int warp = (int)blockIdx.x * STREAM_WARPS + (threadIdx.x >> 5);
  EpiPower<C> epi;
  epi.dinv = dinv;
  epi.y = y;
  epi.f = (C)a.scal[SC_F];
  epi.ss = 0.0;
  stream_rows<V, C, C>(n, warp < warps ? warp : ranges, warps, ranges, part, row_ptr, col, val, x,
                       sh.prod[threadIdx.x >> 5], epi);
  power_finish<C>(a, epi.ss, 0.0, red, last_step);
}

// one row of a step by a warp: y_row = D^-1 (A x)_row (FP64: times f); lane
// q < B adds the square of its component to ss and, if asked, of x to xx
template <class C, class V, int B>
__device__ __forceinline__ void power_row(int row, int lane, const int* ptr, const int* col, const Vals<C, V, B>& A,
                                          const C* dinv, const C* x, C* y, C f, const PowerScale<C>& sc, bool want_xx,
                                          double& ss, double& xx) {
  C dq[B], s[B];
#pragma unroll
  for (int j = 0; j < B; j++) {
    dq[j] = lane < B ? dinv[(int64_t)row * B * B + B * lane + j] : C(0);
    s[j] = C(0);
  }
  for (int k = ptr[row] + lane; k < ptr[row + 1]; k += 32) {
    const int c = __ldg(col + k);
    C v[B * B], g[B];
    A.block(k, v);
#pragma unroll
    for (int j = 0; j < B; j++) g[j] = sc(x[(int64_t)B * c + j]);
#pragma unroll
    for (int q = 0; q < B; q++)
#pragma unroll
      for (int j = 0; j < B; j++) s[q] += v[B * q + j] * g[j];
  }
#pragma unroll
  for (int q = 0; q < B; q++)
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
  if (lane >= B) return;
  C t = C(0);
#pragma unroll
  for (int j = 0; j < B; j++) t += dq[j] * s[j];
  if (sizeof(C) == 8) t *= f;
  y[(int64_t)B * row + lane] = t;
  ss += (double)t * (double)t;
  if (want_xx) {
    const double xv = (double)sc(x[(int64_t)B * row + lane]);
    xx += xv * xv;
  }
}

// coarse levels, and level 0 in FP32: a warp per row, rows strided over at
// most POWER_BLOCKS_PER_SM blocks per SM (a partial sum and a ticket each).
// Level 0 of Cook P2 45x41x7: 45 us, of which the blocks are 18 us at the copy
// rate (before 100 us in three kernels); a coarse level's 14 us are latency.
constexpr int POWER_BLOCKS_PER_SM = 8;
template <class C, class V, int B>
__global__ void __launch_bounds__(256) k_amg_power(int n, const int* __restrict__ ptr, const int* __restrict__ col,
                                                   Vals<C, V, B> A, const C* __restrict__ dinv,
                                                   const C* __restrict__ x, C* __restrict__ y, PowerArgs a,
                                                   bool last_step) {
  __shared__ double red[32];
  const double f = a.scal[SC_F];
  const PowerScale<C> sc(f);
  const int lane = threadIdx.x & 31, nw = (int)((gridDim.x * blockDim.x) >> 5);
  double ss = 0.0, xx = 0.0;
  for (int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); row < n; row += nw)
    power_row<C, V, B>(row, lane, ptr, col, A, dinv, x, y, (C)f, sc, sizeof(C) == 4 && last_step, ss, xx);
  power_finish<C>(a, ss, xx, red, last_step);
}

// The smallest FP32 levels: all 15 steps in one block, while its one SM is
// done before 15 launches are.  The whole setup, in one block and as launches,
// for levels of 144, 250, 455, 884, 1,794 and 2,113 blocks: 391 and 440 us, 443
// and 478, 563 and 609, 663 and 696 (884 blocks of another mesh 1.19 and 1.23
// ms), 0.98 and 0.95 ms, 1.40 and 1.35 ms.  In FP64 the launches win throughout
// (144: 748 and 649 us, 250: 952 and 666, 884: 2.38 and 2.12 ms).
constexpr int AMG_POWER_SMALL = 1024;  // blocks of the level
__global__ void __launch_bounds__(512) k_amg_power_small(int n, int steps, const int* __restrict__ ptr,
                                                         const int* __restrict__ col, Vals<float, float, AMG_NS> A,
                                                         const float* __restrict__ dinv, float* x, float* y, PowerArgs a) {
  __shared__ double red[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int it = 0; it < steps; it++) {
    const double f = ((volatile double*)a.scal)[SC_F];
    const PowerScale<float> sc(f);
    const bool last = it == steps - 1;
    double ss = 0.0, xx = 0.0;
    for (int row = wid; row < n; row += nw)
      power_row<float, float, AMG_NS>(row, lane, ptr, col, A, dinv, x, y, (float)f, sc, last, ss, xx);
    ss = power_block_sum(ss, red);  // (its barriers order this step's rows before the next one's)
    xx = power_block_sum(xx, red);
    if (threadIdx.x == 0) power_result<float>(a, ss, xx, last);
    __syncthreads();
    float* t = x;
    x = y;
    y = t;
  }
}

__global__ void k_amg_to_f32(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}

// Once per mesh: the blocks of every fine row grouped by the aggregate of
// their column, one list per P entry (pk[pk_ptr[q].x .. pk_ptr[q].y)), and
// the place of each P entry in R = P^T.
__global__ void k_amg_plists(int n, const int* __restrict__ ptr, const int* __restrict__ col,
                             const int* __restrict__ agg, const int* __restrict__ pptr, const int* __restrict__ pcol,
                             int2* __restrict__ pk_ptr, int* __restrict__ pk) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int o = ptr[i];
  for (int q = pptr[i]; q < pptr[i + 1]; q++) {
    const int a = pcol[q], o0 = o;
    for (int k = ptr[i]; k < ptr[i + 1]; k++)
      if (agg[col[k]] == a) pk[o++] = k;
    pk_ptr[q] = make_int2(o0, o);
  }
}
__global__ void k_amg_rpos(int64_t nnzr, const int* __restrict__ rsrc, int* __restrict__ rpos) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < nnzr) rpos[rsrc[s]] = (int)s;
}

// P entry q = (row i, aggregate a): [agg(i) = a] T_i - omega sum over the row's
// blocks k with agg(col k) = a of (D_i^-1 A_k) T_col(k), k ascending.  B
// threads per entry, one row each: the blocks come from the entry's list (a
// thread per entry that scanned its whole row took 632 us for 629k entries),
// the block and T's rows are shared by neighbouring threads.  Also writes the
// V-cycle's tiled copy pt and the transpose R (their own kernels took 30 and
// 58 us).  Cook P2 45x41x7: level 0 176 us (before 447), level 1 119.
template <class C, class V, int B>
__global__ void __launch_bounds__(B == 3 ? 192 : 64) k_amg_pvals(int64_t nnzp, const int* __restrict__ prow,
                                                   const int* __restrict__ pcol, const int2* __restrict__ pk_ptr,
                                                   const int* __restrict__ pk, const int* __restrict__ col,
                                                   Vals<C, V, B> A, const int* __restrict__ agg,
                                                   const C* __restrict__ dinv, const C* __restrict__ tnode,
                                                   const double* __restrict__ scal, const int* __restrict__ rpos,
                                                   C* __restrict__ p, C* __restrict__ pt, C* __restrict__ rv) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t q = t / B;
  const int r = (int)(t % B);
  if (q >= nnzp) return;
  const int i = prow[q];
  const C omega = (C)scal[SC_OMEGA];
  const bool own = agg[i] == pcol[q];
  C acc[AMG_NS], d[B];
#pragma unroll
  for (int c = 0; c < AMG_NS; c++) acc[c] = own ? tnode[((int64_t)i * B + r) * AMG_NS + c] : C(0);
#pragma unroll
  for (int l = 0; l < B; l++) d[l] = dinv[((int64_t)i * B + r) * B + l];
  const int2 lst = pk_ptr[q];
  int k = lst.x < lst.y ? pk[lst.x] : 0, j = lst.x < lst.y ? col[k] : 0;
  for (int e = lst.x; e < lst.y; e++) {
    const C* T = tnode + (int64_t)j * B * AMG_NS;
    C av[B * B], da[B];
    A.block(k, av);
    if (e + 1 < lst.y) {
      k = pk[e + 1];
      j = col[k];
    }
#pragma unroll
    for (int c = 0; c < B; c++) {
      C v = C(0);
#pragma unroll
      for (int l = 0; l < B; l++) v += d[l] * av[B * l + c];
      da[c] = v;
    }
#pragma unroll
    for (int c = 0; c < AMG_NS; c++) {
      C v = C(0);
#pragma unroll
      for (int l = 0; l < B; l++) v += da[l] * T[AMG_NS * l + c];
      acc[c] -= omega * v;
    }
  }
  const int64_t rp = (int64_t)rpos[q] * B * AMG_NS;
#pragma unroll
  for (int c = 0; c < AMG_NS; c++) {
    p[q * B * AMG_NS + AMG_NS * r + c] = acc[c];
    pt[tix<B * AMG_NS>(q, AMG_NS * r + c)] = acc[c];
    rv[rp + B * c + r] = acc[c];
  }
}

// place of c among the m ascending values of list, -1 if absent
__device__ __forceinline__ int find_sorted(const int* list, int m, int c) {
  int lo = 0;
  for (int len = m; len > 0;) {  // first place whose value is not below c
    const int half = len >> 1;
    const bool below = list[lo + half] < c;
    lo = below ? lo + half + 1 : lo;
    len = below ? len - half - 1 : half;
  }
  return lo < m && list[lo] == c ? lo : -1;
}

// Once per mesh: the place in its A P row of every product A_k P_q of a fine
// row (k in order, then q in P row col k).
__global__ void k_amg_apidx(int n, const int* __restrict__ ptr, const int* __restrict__ col,
                            const int* __restrict__ pptr, const int* __restrict__ pcol, const int* __restrict__ apptr,
                            const int* __restrict__ apcol, const int64_t* __restrict__ off, int* __restrict__ idx) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  int64_t o = off[i];
  const int a0 = apptr[i], m = apptr[i + 1] - a0;
  for (int k = ptr[i]; k < ptr[i + 1]; k++) {
    const int j = col[k], q0 = pptr[j], q1 = pptr[j + 1];
    for (int q = q0 + lane; q < q1; q += 32) idx[o + (q - q0)] = find_sorted(apcol + a0, m, pcol[q]);
    o += q1 - q0;
  }
}
// Once per mesh: the products P_q^T (A P)_e of every coarse entry (q of P^T row
// a in order, e the entry of q's node in the coarse column), one list per
// entry, and the entry's row.  A warp per coarse row counts, sums the counts
// and fills; the entries of one A P row have distinct places.
__global__ void k_amg_raplists(int nc, const int* __restrict__ cptr, const int* __restrict__ ccol,
                               const int* __restrict__ rptr, const int* __restrict__ rcol,
                               const int* __restrict__ rsrc, const int* __restrict__ apptr,
                               const int* __restrict__ apcol, const int64_t* __restrict__ raoff,
                               int64_t* lend, int* crow, int2* __restrict__ list) {  // (no list: the rows alone)
  const int a = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (a >= nc) return;
  const int c0 = cptr[a], m = cptr[a + 1] - c0;
  for (int t = lane; t < m; t += 32) {
    lend[c0 + t] = 0;
    crow[c0 + t] = a;
  }
  if (!list) return;
  __syncwarp();
  for (int pass = 0; pass < 2; pass++) {
    for (int s = rptr[a]; s < rptr[a + 1]; s++) {
      const int e1 = apptr[rcol[s] + 1];
      for (int e = apptr[rcol[s]] + lane; e < e1; e += 32) {
        const int pos = find_sorted(ccol + c0, m, apcol[e]);
        if (pos < 0) continue;
        const int64_t o = lend[c0 + pos]++;
        if (pass) list[o] = make_int2(rsrc[s], e);
      }
      __syncwarp();
    }
    if (pass) break;
    int64_t base = raoff[a];  // counts -> starts; the fill leaves the ends
    for (int t0 = 0; t0 < m; t0 += 32) {
      const int64_t v = t0 + lane < m ? lend[c0 + t0 + lane] : 0;
      int64_t inc = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      if (t0 + lane < m) lend[c0 + t0 + lane] = base + inc - v;
      base += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncwarp();
  }
}

// A P, one warp per fine row: the row's blocks A_k (staged in shared memory,
// 32 at a time) times the P rows of their columns, five P entries of a row at
// a time (lane 6 g + c: entry g, column c), added up in shared memory at the
// product's place in the A P row (a list made once per mesh: searched for
// here, the places took more instructions than the products).  Rows longer than
// AMG_CHUNK entries are taken in chunks.  Without the list (LIST false) the
// place is searched, to the same sums.  The entries of one P row have
// distinct places and block k + 1 follows block k after a warp barrier: no
// atomics, a fixed order.  Bound by the
// FP32 and shared-memory instructions of the products: about 500 us on level 0
// of Cook P2 45x41x7 (113k rows, 1.9 M entries).  Before, a thread per output
// entry that searched the P rows of all the row's columns: 638 us there, and
// 204 us on the next level, now 51.
constexpr int AMG_CHUNK = 64;
template <class C, int B>
struct ApShared {
  C acc[AMG_CHUNK * B * AMG_NS];
  C a[32][B * B];
};
template <class C, int B>
__host__ __device__ constexpr int ap_warps() { return B == 3 && sizeof(C) == 4 ? 8 : 4; }

template <class C, class V, int B, bool LIST>
__global__ void __launch_bounds__(32 * ap_warps<C, B>())
    k_amg_ap(int n, const int* __restrict__ ptr, const int* __restrict__ col, Vals<C, V, B> A,
             const int* __restrict__ pptr, const int* __restrict__ pcol, const C* __restrict__ p,
             const int* __restrict__ apptr, const int* __restrict__ apcol, const int64_t* __restrict__ apoff,
             const int* __restrict__ apidx, C* __restrict__ ap) {
  constexpr int BN = B * AMG_NS;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  ApShared<C, B>& sh = reinterpret_cast<ApShared<C, B>*>(smraw)[wid];
  const int i = blockIdx.x * ap_warps<C, B>() + wid;
  if (i >= n) return;
  const int g = lane / AMG_NS, c = lane % AMG_NS;
  const int ks = ptr[i], ke = ptr[i + 1], a0 = apptr[i], ae = apptr[i + 1];
  for (int cb = a0; cb < ae; cb += AMG_CHUNK) {
    const int m = min(AMG_CHUNK, ae - cb);
    const int* ix = LIST ? apidx + apoff[i] : nullptr;  // places of the next block's products
    for (int t = lane; t < m * BN; t += 32) sh.acc[t] = C(0);
    for (int k0 = ks; k0 < ke; k0 += 32) {
      const int cnt = min(32, ke - k0);
      int q0 = 0, q1 = 0;
      if (lane < cnt) {
        const int j = col[k0 + lane];
        q0 = pptr[j];
        q1 = pptr[j + 1];
        C av[B * B];
        A.block(k0 + lane, av);
#pragma unroll
        for (int t = 0; t < B * B; t++) sh.a[lane][t] = av[t];
      }
      __syncwarp();
      for (int kk = 0; kk < cnt; kk++) {
        const int qa = __shfl_sync(0xffffffffu, q0, kk), len = __shfl_sync(0xffffffffu, q1, kk) - qa;
        if (g < 5)
          for (int u = g; u < len; u += 5) {
            const int e = (LIST ? ix[u] : find_sorted(apcol + a0, ae - a0, pcol[qa + u])) - (cb - a0);
            const C* P = p + (int64_t)(qa + u) * BN + c;
            C pv[B];
#pragma unroll
            for (int l = 0; l < B; l++) pv[l] = P[AMG_NS * l];
            if (e >= 0 && e < m) {
              C* o = sh.acc + e * BN + c;
#pragma unroll
              for (int r = 0; r < B; r++) {
                C s = C(0);
#pragma unroll
                for (int l = 0; l < B; l++) s += sh.a[kk][B * r + l] * pv[l];
                o[AMG_NS * r] += s;
              }
            }
          }
        if (LIST) ix += len;
        __syncwarp();
      }
    }
    for (int t = lane; t < m * BN; t += 32) ap[(int64_t)cb * BN + t] = sh.acc[t];
    __syncwarp();
  }
}

// Coarse operator: entry e = (a, b) is the sum over its list (q ascending) of
// P_q^T (A P)_(node of q, b); absent components get a unit diagonal.  B = 3
// (level 0, many entries with some hundred products each): six threads per
// entry, one row each, the A P values shared by neighbouring threads.  B = 6
// (few entries, long lists, bound by the latency of the loads): 36 threads, one
// value each, eight products in flight.  404 us on level 0 of Cook P2 45x41x7
// and 167 us on level 1 (a thread per entry that searched the
// A P rows of all the row's nodes: 979 and 849 us).  Without the list (LIST
// false) the A P rows are searched, to the same sums.
template <class C, int B, bool LIST>
__global__ void __launch_bounds__(B == 3 ? 192 : 64)
    k_amg_rap(int64_t nnzc, const int* __restrict__ crow, const int* __restrict__ ccol,
              const int64_t* __restrict__ lend, const int64_t* __restrict__ raoff, const int2* __restrict__ list,
              const int* __restrict__ rptr, const int* __restrict__ rcol, const int* __restrict__ rsrc,
              const int* __restrict__ apptr, const int* __restrict__ apcol, const C* __restrict__ p, const C* __restrict__ ap, const unsigned char* __restrict__ cabsent,
              C* __restrict__ out) {
  constexpr int BN = B * AMG_NS, NN = AMG_NS * AMG_NS;
  constexpr int PER = B == 3 ? AMG_NS : 1, TPE = NN / PER;  // values per thread, threads per entry
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t e = t / TPE;
  if (e >= nnzc) return;
  const int u = (int)(t % TPE), r = PER == 1 ? u / AMG_NS : u, cc = PER == 1 ? u % AMG_NS : 0;
  const int a = crow[e];
  C acc[PER];
#pragma unroll
  for (int c = 0; c < PER; c++) acc[c] = C(0);
  constexpr int U = B == 3 ? 2 : (sizeof(C) == 4 ? 8 : 4);  // products in flight
  auto add = [&](const C (&P)[B], const C (&Q)[B][PER]) {
#pragma unroll
    for (int c = 0; c < PER; c++) {
      C v = C(0);
#pragma unroll
      for (int k = 0; k < B; k++) v += P[k] * Q[k][c];
      acc[c] += v;
    }
  };
  auto load = [&](int2 it, C (&P)[B], C (&Q)[B][PER]) {
    const C* pp = p + (int64_t)it.x * BN + r;
    const C* qq = ap + (int64_t)it.y * BN + cc;
#pragma unroll
    for (int k = 0; k < B; k++) {
      P[k] = __ldg(pp + AMG_NS * k);
#pragma unroll
      for (int c = 0; c < PER; c++) Q[k][c] = __ldg(qq + AMG_NS * k + c);
    }
  };
  if constexpr (LIST) {
    const int64_t l1 = lend[e];
    int64_t l = e > 0 && crow[e - 1] == a ? lend[e - 1] : raoff[a];
    for (; l + U <= l1; l += U) {
      C P[U][B], Q[U][B][PER];
#pragma unroll
      for (int w = 0; w < U; w++) load(list[l + w], P[w], Q[w]);
#pragma unroll
      for (int w = 0; w < U; w++) add(P[w], Q[w]);
    }
    for (; l < l1; l++) {
      C P[B], Q[B][PER];
      load(list[l], P, Q);
      add(P, Q);
    }
  } else {
    for (int s = rptr[a]; s < rptr[a + 1]; s++) {
      const int f0 = apptr[rcol[s]], pos = find_sorted(apcol + f0, apptr[rcol[s] + 1] - f0, ccol[e]);
      if (pos < 0) continue;
      C P[B], Q[B][PER];
      load(make_int2(rsrc[s], f0 + pos), P, Q);
      add(P, Q);
    }
  }
  const bool unit = ccol[e] == a && ((cabsent[a] >> r) & 1u);
#pragma unroll
  for (int c = 0; c < PER; c++) out[e * NN + AMG_NS * r + cc + c] = unit && cc + c == r ? C(1) : acc[c];
}

// dense inverse of the coarsest operator (N <= 96): one block, Gauss-Jordan
// in place in shared memory with partial pivoting (first maximal pivot on
// ties, found by one warp on the bit patterns), FP64; the row exchanges
// become column exchanges of the inverse.  The FP64 pipe bounds it: N^2
// products per column instead of the 2 N^2 of [A | I] (N = 24: 41 us;
// N = 66 took 525 us as [A | I] with a serial pivot search).
template <class C, class V, int B>
__global__ void __launch_bounds__(1024) k_amg_dense_inverse(int n, const int* __restrict__ ptr,
                                                            const int* __restrict__ col, Vals<C, V, B> A,
                                                            double* __restrict__ inv, float* __restrict__ inv32) {
  extern __shared__ double sm[];
  const int N = n * B;
  double* M = sm;
  double* fac = sm + N * N;       // column c before the elimination step
  double* row = fac + N;          // row c after scaling
  __shared__ int s_piv[AMG_DENSE_MAX];
  __shared__ double s_rp;
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) M[t] = 0.0;
  __syncthreads();
  for (int a = threadIdx.x; a < n; a += blockDim.x)
    for (int k = ptr[a]; k < ptr[a + 1]; k++)
      for (int r = 0; r < B; r++)
        for (int c = 0; c < B; c++) M[(B * a + r) * N + B * col[k] + c] = (double)A(k, B * r + c);
  __syncthreads();
  for (int c = 0; c < N; c++) {
    if (threadIdx.x < 32) {
      unsigned long long best = 0;
      int p = c;
      for (int r = c + (int)threadIdx.x; r < N; r += 32) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(M[r * N + c]) & 0x7fffffffffffffffULL;
        if (b > best) {
          best = b;
          p = r;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long b = __shfl_xor_sync(0xffffffffu, best, o);
        const int q = __shfl_xor_sync(0xffffffffu, p, o);
        if (b > best || (b == best && q < p)) {
          best = b;
          p = q;
        }
      }
      if (threadIdx.x == 0) {
        s_piv[c] = p;
        s_rp = 1.0 / M[p * N + c];
      }
    }
    __syncthreads();
    const int p = s_piv[c];
    const double rp = s_rp;
    // row c <- row p / pivot (with 1 in column c), row p <- row c
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      const double vp = M[p * N + j], vc = M[c * N + j];
      row[j] = (j == c ? 1.0 : vp) * rp;
      if (p != c) M[p * N + j] = vc;
    }
    __syncthreads();
    for (int r = threadIdx.x; r < N; r += blockDim.x) fac[r] = r == c ? 0.0 : M[r * N + c];
    __syncthreads();
    for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
      const int r = t / N, j = t - r * N;
      M[t] = r == c ? row[j] : (j == c ? 0.0 : M[t]) - fac[r] * row[j];
    }
    __syncthreads();
  }
  for (int c = N - 1; c >= 0; c--) {
    const int p = s_piv[c];
    if (p != c)
      for (int r = threadIdx.x; r < N; r += blockDim.x) {
        const double t = M[r * N + c];
        M[r * N + c] = M[r * N + p];
        M[r * N + p] = t;
      }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
    inv[t] = M[t];
    if (inv32) inv32[t] = (float)M[t];
  }
}

// ---------------------------------------------------------------- V-cycle kernels
// One Chebyshev step of level l, fused (row i of n block rows, B components):
//   t = (A g)_i; x_i = (setx ? 0 : x_i) + cx g_i; r_i -= t;
//   dout_i = c1 g_i + c2 D_i^-1 r_i; final: x_i += dout_i.
// One warp per block row, one lane per block; level 0 reads the tangent
// in its tiled layout.
enum { VC_SETX = 1, VC_FINAL = 2, VC_KEEPX = 4, VC_START = 8 };


// Level-0 Chebyshev step: the streamed product of fe_stream.cuh with the row
// updates as its epilogue; a window's g, r, x and block-Jacobi inverses are
// copied to shared memory while its tiles are multiplied.  Five blocks per SM
// (96 registers) in FP32: with six the operands spill (48x48x8: 312 against
// 278 us per V-cycle).
template <class T>
__host__ __device__ constexpr int cheb0_blocks_per_sm() { return sizeof(T) == 8 ? 3 : 5; }

template <class T>
struct ChebStage {  // operands of up to 16 rows of a window
  T g[48], r[48], x[48], d[144];
};

template <class T>
struct EpiCheb {
  const T* dinv;
  const T* g;
  T* x;
  T* r;
  T* dout;
  T cx, k1, k2;
  int flags;
  ChebStage<T>* st;
  T gi[3], ri[3], xo[3], di[9];
  // copies a window's rows into the stage while its tiles are multiplied
  __device__ __forceinline__ void prefetch(int r0, int rb, int lane) {
    const int m = min(16, rb - r0);
    const int64_t o = 3 * (int64_t)r0;
    for (int i = lane; i < 3 * m; i += 32) {
      cp_async(st->g + i, g + o + i);
      cp_async(st->r + i, r + o + i);
      if (!(flags & (VC_KEEPX | VC_SETX))) cp_async(st->x + i, x + o + i);
    }
    if (dout)
      for (int i = lane; i < 9 * m; i += 32) cp_async(st->d + i, dinv + 3 * o + i);
  }
  __device__ __forceinline__ void load(int r0, int i0, int nd, int lane) {
    cp_async_wait();
    __syncwarp();  // (a lane reads what other lanes copied)
    if (lane >= nd) return;
    const bool in = i0 + lane < 16;
    const int64_t o = 3 * (int64_t)(r0 + lane);
    const int i = i0 + lane;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      gi[q] = in ? st->g[3 * i + q] : g[o + q];
      ri[q] = in ? st->r[3 * i + q] : r[o + q];
      xo[q] = (flags & (VC_KEEPX | VC_SETX)) ? T(0) : (in ? st->x[3 * i + q] : x[o + q]);
    }
    if (dout)
#pragma unroll
      for (int q = 0; q < 9; q++) di[q] = in ? st->d[9 * i + q] : dinv[3 * o + q];
  }
  __device__ __forceinline__ void finish(int row, const T (&s)[3]) {
    const int64_t o = 3 * (int64_t)row;
    T rn[3], xi[3];
#pragma unroll
    for (int q = 0; q < 3; q++) {
      rn[q] = ri[q] - s[q];
      r[o + q] = rn[q];
      xi[q] = xo[q] + cx * gi[q];
    }
    if (dout) {
#pragma unroll
      for (int q = 0; q < 3; q++) {
        T t = T(0);
#pragma unroll
        for (int j = 0; j < 3; j++) t += di[3 * q + j] * rn[j];
        const T dn = k1 * gi[q] + k2 * t;
        if (flags & VC_FINAL) xi[q] += dn;  // (the final direction is in x already)
        else dout[o + q] = dn;
      }
    }
    if (!(flags & VC_KEEPX))
#pragma unroll
      for (int q = 0; q < 3; q++) x[o + q] = xi[q];
  }
};

template <class V, class T>
__global__ void __launch_bounds__(STREAM_THREADS, cheb0_blocks_per_sm<T>())
    k_vc_cheb0(int n, int warps, int ranges, const int* __restrict__ part, const int* __restrict__ row_ptr,
               const int* __restrict__ col, const V* __restrict__ val, const T* __restrict__ dinv,
               const T* __restrict__ g, T* __restrict__ x, T* __restrict__ r, T* __restrict__ dout, T cx,
               const T* __restrict__ coef, int flags) {
  __shared__ StreamShared<T> sh;
  __shared__ __align__(16) ChebStage<T> stage[STREAM_WARPS];
  const int warp = (int)blockIdx.x * STREAM_WARPS + (threadIdx.x >> 5);
  if (warp >= warps) return;
  EpiCheb<T> epi;
  epi.st = &stage[threadIdx.x >> 5];
  epi.dinv = dinv;
  epi.g = g;
  epi.x = x;
  epi.r = r;
  epi.dout = dout;
  epi.cx = cx;
  epi.k1 = (flags & VC_START) ? T(0) : coef[1];
  epi.k2 = (flags & VC_START) ? coef[0] : coef[2];
  epi.flags = flags;
  stream_rows<V, T, T>(n, warp, warps, ranges, part, row_ptr, col, val, g, sh.prod[threadIdx.x >> 5], epi);
}

// The same step for the largest FP32 levels: a warp takes groups of 16
// consecutive block rows and walks their (contiguous) blocks in chunks of 32,
// one block per lane, forming the row sums by a segmented scan across the
// lanes and carrying a row's partial sum into the next chunk; values, column
// indices and the gather of g run ahead.  A row's sum goes to shared memory
// when its last block is reached; the group's 16 Chebyshev row updates run
// together after its last chunk, lane i on row i, with the rows' g, r, x and
// block-Jacobi inverse loaded when the group starts.
//
// The loads of a group never wait for a phase of row sums, which is worth 7%
// of the V-cycle where HBM bounds it, but groups of 16 rows must fill the
// wave several times: per V-cycle, scan against window form, FP32: Cook P2
// 64x64x8 (4.8 groups per warp) 417 and 446 us, 48x48x8 (2.7) 288 and 278,
// 30x26x6 (one) 113 and 87, cardiac shell 72 and 71; FP64: 2,420 and 1,688,
// 1,518 and 995, 609 and 332, 363 and 316 us (the scan's adds, 15 per block).
constexpr int VC_RPW = 16;

template <class V, class T>
__device__ __forceinline__ void vc_load_chunk(const int* __restrict__ col, const V* __restrict__ val, int64_t k,
                                              int64_t kend, int& c, T (&v)[9]) {
  if (k < kend) {
    c = __ldg(col + k);
#pragma unroll
    for (int t = 0; t < 9; t++) v[t] = ldt<T, V>(val + tix<9>(k, t));
  } else {
    c = -1;
#pragma unroll
    for (int t = 0; t < 9; t++) v[t] = T(0);
  }
}

template <class T>
__device__ __forceinline__ void vc_load_g(const T* __restrict__ g, int c, T (&x)[3], int n) {
  const int64_t cc = c >= 0 ? fe_idx(c, n) : 0;
#pragma unroll
  for (int j = 0; j < 3; j++) x[j] = c >= 0 ? g[3 * cc + j] : T(0);
}

template <class V, class T>
__global__ void __launch_bounds__(256) k_vc_cheb0_scan(int n, const int* __restrict__ row_ptr, const int* __restrict__ col,
                                                  const V* __restrict__ val, const T* __restrict__ dinv,
                                                  const T* __restrict__ g, T* __restrict__ x, T* __restrict__ r,
                                                  T* __restrict__ dout, T cx, const T* __restrict__ coef,
                                                  int flags) {
  __shared__ T rsum[8][VC_RPW][3];  // row sums of each warp's current group
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool wx = !(flags & VC_KEEPX), rx = wx && !(flags & VC_SETX);
  const int ngroups = (n + VC_RPW - 1) / VC_RPW;
  const int nwarps = (int)(((int64_t)gridDim.x * blockDim.x) >> 5);
  for (int grp = (int)((((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5)); grp < ngroups; grp += nwarps) {
    const int r0 = grp * VC_RPW;
    const int nr = min(VC_RPW, n - r0);
    const int rpl = lane < nr ? __ldg(row_ptr + r0 + lane) : INT_MAX;  // start of row r0 + lane
    const int kstart = __shfl_sync(0xffffffffu, rpl, 0);
    const int kend = __ldg(row_ptr + r0 + nr);
    // this lane's row of the group (lane < nr): its update operands, loaded now
    T gi[3] = {T(0), T(0), T(0)}, ri[3] = {T(0), T(0), T(0)}, xo[3] = {T(0), T(0), T(0)}, di[9];
#pragma unroll
    for (int q = 0; q < 9; q++) di[q] = T(0);
    if (lane < nr) {
      const int64_t o = 3 * (int64_t)(r0 + lane);
#pragma unroll
      for (int q = 0; q < 3; q++) {
        gi[q] = g[o + q];
        ri[q] = r[o + q];
        if (rx) xo[q] = x[o + q];
      }
      if (dout)
#pragma unroll
        for (int q = 0; q < 9; q++) di[q] = dinv[9 * (int64_t)(r0 + lane) + q];
    }
    int c0, c1;
    T v0[9], v1[9];
    vc_load_chunk<V, T>(col, val, (int64_t)kstart + lane, kend, c0, v0);
    vc_load_chunk<V, T>(col, val, (int64_t)kstart + 32 + lane, kend, c1, v1);
    T xa[3];
    vc_load_g<T>(g, c0, xa, n);
    T carry[3] = {T(0), T(0), T(0)};
    int rowbase = r0 - 1;
    for (int kc = kstart; kc < kend; kc += 32) {
      int c2;
      T v2[9];
      vc_load_chunk<V, T>(col, val, (int64_t)kc + 64 + lane, kend, c2, v2);
      T xb[3];
      vc_load_g<T>(g, c1, xb, n);
      T p[3] = {T(0), T(0), T(0)};
      if (c0 >= 0)
#pragma unroll
        for (int q = 0; q < 3; q++) p[q] = v0[3 * q] * xa[0] + v0[3 * q + 1] * xa[1] + v0[3 * q + 2] * xa[2];
      const unsigned bit = (rpl >= kc && rpl - kc < 32) ? (1u << (rpl - kc)) : 0u;
      const unsigned heads = __reduce_or_sync(0xffffffffu, bit);
      const unsigned below = heads & (0xffffffffu >> (31 - lane));
      const int sstart = below ? 31 - __clz(below) : -1;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        T t[3];
#pragma unroll
        for (int q = 0; q < 3; q++) t[q] = __shfl_up_sync(0xffffffffu, p[q], off);
        if (lane >= off && lane - off >= sstart)
#pragma unroll
          for (int q = 0; q < 3; q++) p[q] += t[q];
      }
      const int nvalid = min(32, kend - kc);
      const bool cont = nvalid == 32 && kc + 32 < kend && !__any_sync(0xffffffffu, rpl == kc + 32);
      const bool tail = lane < nvalid && ((lane < 31 && ((heads >> (lane + 1)) & 1u)) || (lane == nvalid - 1 && !cont));
      if (tail) {
        const int row = rowbase + __popc(below);
        const bool add = sstart < 0;
#pragma unroll
        for (int q = 0; q < 3; q++) rsum[wid][row - r0][q] = p[q] + (add ? carry[q] : T(0));
      }
      T l[3];
#pragma unroll
      for (int q = 0; q < 3; q++) l[q] = __shfl_sync(0xffffffffu, p[q], 31);
      if (cont) {
        const bool whole = heads == 0u;  // lane 31's segment started before this chunk
#pragma unroll
        for (int q = 0; q < 3; q++) carry[q] = l[q] + (whole ? carry[q] : T(0));
      } else {
#pragma unroll
        for (int q = 0; q < 3; q++) carry[q] = T(0);
      }
      rowbase += __popc(heads);
      c0 = c1;
      c1 = c2;
#pragma unroll
      for (int t = 0; t < 9; t++) {
        v0[t] = v1[t];
        v1[t] = v2[t];
      }
#pragma unroll
      for (int j = 0; j < 3; j++) xa[j] = xb[j];
    }
    __syncwarp();
    if (lane < nr) {  // the group's row updates (cheb_rows' arithmetic, operands preloaded)
      const int64_t row = r0 + lane, o = 3 * row;
      T rn[3], xi[3];
#pragma unroll
      for (int q = 0; q < 3; q++) {
        rn[q] = ri[q] - rsum[wid][lane][q];
        r[o + q] = rn[q];
        xi[q] = xo[q] + cx * gi[q];
      }
      if (dout) {
        const T k1 = (flags & VC_START) ? T(0) : coef[1];
        const T k2 = (flags & VC_START) ? coef[0] : coef[2];
#pragma unroll
        for (int q = 0; q < 3; q++) {
          T t = T(0);
#pragma unroll
          for (int jj = 0; jj < 3; jj++) t += di[3 * q + jj] * rn[jj];
          const T dn = k1 * gi[q] + k2 * t;
          dout[o + q] = dn;
          if (flags & VC_FINAL) xi[q] += dn;
        }
      }
      if (wx)
#pragma unroll
        for (int q = 0; q < 3; q++) x[o + q] = xi[q];
    }
    __syncwarp();
  }
}

// Chebyshev step of a coarse level, one block row per warp (coarse rows
// are few and long), one lane per block; a lane reads its 6x6 block
// (block-major, from a device allocation, so 16-byte aligned) with 16-byte
// loads: nine load instructions in FP32 instead of 36.  Device function of
// warp-uniform `row` (< n): the kernel below runs it for its warp's row, the
// fused bottom of the V-cycle (k_vc_bottom) for rows strided over its warps;
// both sum in the same order, so their results are identical.  Vectors are
// read with plain loads: in k_vc_bottom they were written by the same block.
template <class T, int B>
__device__ __forceinline__ void vc_cheb_row(int row, int lane, int n, const int* ptr, const int* col, const T* val,
                                            const T* dinv, const T* g, T* x, T* r, T* dout, T cx, const T* coef,
                                            int flags) {
  // lane q < B updates component q of the row (cheb_rows' arithmetic); its
  // operands are loaded before the row's products, so their latency overlaps
  const bool wx = !(flags & VC_KEEPX), rx = wx && !(flags & VC_SETX);
  const int64_t o = (int64_t)B * row;
  T gq = T(0), rq = T(0), xq = T(0), dq[B];
#pragma unroll
  for (int j = 0; j < B; j++) dq[j] = T(0);
  if (lane < B) {
    gq = g[o + lane];
    rq = r[o + lane];
    if (rx) xq = x[o + lane];
    if (dout)
#pragma unroll
      for (int j = 0; j < B; j++) dq[j] = dinv[(int64_t)row * B * B + B * lane + j];
  }
  T s[B];
#pragma unroll
  for (int q = 0; q < B; q++) s[q] = T(0);
  for (int k = ptr[row] + lane; k < ptr[row + 1]; k += 32) {
    const int c = fe_idx(__ldg(col + k), n);
    T v[B * B];
    load_block6<T>(val, k, v);
    T gv[B];
#pragma unroll
    for (int j = 0; j < B; j++) gv[j] = g[(int64_t)B * c + j];
#pragma unroll
    for (int q = 0; q < B; q++)
#pragma unroll
      for (int j = 0; j < B; j++) s[q] += v[B * q + j] * gv[j];
  }
#pragma unroll
  for (int q = 0; q < B; q++)
    for (int off = 16; off > 0; off >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
  // this lane's component of the new residual, then every lane gets all of them
  T sq = T(0);
#pragma unroll
  for (int q = 0; q < B; q++)
    if (q == lane) sq = s[q];
  const T rn_q = rq - sq;
  T rn[B];
#pragma unroll
  for (int j = 0; j < B; j++) rn[j] = __shfl_sync(0xffffffffu, rn_q, j);
  if (lane < B) {
    r[o + lane] = rn_q;
    T xi = xq + cx * gq;
    if (dout) {
      const T c1 = (flags & VC_START) ? T(0) : coef[1];
      const T c2 = (flags & VC_START) ? coef[0] : coef[2];
      T t = T(0);
#pragma unroll
      for (int j = 0; j < B; j++) t += dq[j] * rn[j];
      const T dn = c1 * gq + c2 * t;
      dout[o + lane] = dn;
      if (flags & VC_FINAL) xi += dn;
    }
    if (wx) x[o + lane] = xi;
  }
}

// (FP64, two rows per block: a level of 227 rows spreads over 114 SMs, not 29,
// V-cycles of 12^3 to 30x26x6 meshes are 4-8 % faster; FP32 7.3 us with eight
// rows per block there, 8.1 with two)
template <class T>
constexpr int VC_CHEB_THREADS = sizeof(T) == 8 ? 64 : 256;
template <class T, int B>
__global__ void __launch_bounds__(VC_CHEB_THREADS<T>) k_vc_cheb(int n, const int* __restrict__ ptr, const int* __restrict__ col,
                                                 const T* __restrict__ val, const T* __restrict__ dinv,
                                                 const T* __restrict__ g, T* __restrict__ x, T* __restrict__ r,
                                                 T* __restrict__ dout, T cx, const T* __restrict__ coef,
                                                 int flags) {
  const int row = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  vc_cheb_row<T, B>(row, lane, n, ptr, col, val, dinv, g, x, r, dout, cx, coef, flags);
}

// level-0 start of the pre-smoothing: r = b, d = D^-1 b / theta
template <class T>
__global__ void k_vc_init0(int n, const T* __restrict__ dinv, const double* __restrict__ b, T* __restrict__ r,
                           T* __restrict__ d, const T* __restrict__ coef) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T inv_theta = coef[0];
  T bi[3], di[3];
  for (int q = 0; q < 3; q++) bi[q] = (T)b[3 * (int64_t)i + q];
  for (int q = 0; q < 3; q++) {
    T t = T(0);
    for (int j = 0; j < 3; j++) t += dinv[(int64_t)i * 9 + 3 * q + j] * bi[j];
    di[q] = t * inv_theta;
  }
  for (int q = 0; q < 3; q++) {
    r[3 * (int64_t)i + q] = bi[q];
    d[3 * (int64_t)i + q] = di[q];
  }
}

// restriction to the coarse level (6 components): s = (P^T r)_a;
// coarsest: bout = s; else: rc = s, dc = D_c^-1 s / theta_c.  A block of 128
// threads per coarse row: P^T rows are long (an aggregate's nodes and their
// neighbours, hundreds of blocks at level 0), so a warp per row would leave
// too few warps in flight; the block's partial sums are reduced in a fixed
// order (deterministic).
constexpr int VC_RESTRICT_THREADS = 128;

// thread t's partial sums of coarse row a (entries t, t + 128, ...)
template <class T, int BF>
__device__ __forceinline__ void vc_restrict_part(int a, int t, T (&s)[AMG_NS], const int* rptr, const int* rcol,
                                                 const T* rv, const T* rf, int nfine) {
#pragma unroll
  for (int q = 0; q < AMG_NS; q++) s[q] = T(0);
  for (int k = rptr[a] + t; k < rptr[a + 1]; k += VC_RESTRICT_THREADS) {
    const int i = fe_idx(__ldg(rcol + k), nfine);
    T f[BF];
#pragma unroll
    for (int j = 0; j < BF; j++) f[j] = rf[(int64_t)BF * i + j];
#pragma unroll
    for (int q = 0; q < AMG_NS; q++)
#pragma unroll
      for (int j = 0; j < BF; j++) s[q] += __ldg(rv + (int64_t)k * BF * AMG_NS + BF * q + j) * f[j];
  }
#pragma unroll
  for (int q = 0; q < AMG_NS; q++)
    for (int off = 16; off > 0; off >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
}

// coarse row a from its four warps' sums sh[w][q] (one thread)
template <class T>
__device__ __forceinline__ void vc_restrict_finish(int a, const T (*sh)[AMG_NS], const T* dinvc, T* rc, T* dc,
                                                   const T* coefc) {
  T s[AMG_NS];
#pragma unroll
  for (int q = 0; q < AMG_NS; q++) s[q] = (sh[0][q] + sh[1][q]) + (sh[2][q] + sh[3][q]);
  const int64_t o = (int64_t)AMG_NS * a;
#pragma unroll
  for (int q = 0; q < AMG_NS; q++) rc[o + q] = s[q];
  if (dc) {
    const T inv_theta = coefc[0];
#pragma unroll
    for (int q = 0; q < AMG_NS; q++) {
      T t = T(0);
#pragma unroll
      for (int j = 0; j < AMG_NS; j++) t += dinvc[(int64_t)a * AMG_NS * AMG_NS + AMG_NS * q + j] * s[j];
      dc[o + q] = t * inv_theta;
    }
  }
}

template <class T, int BF>
__global__ void __launch_bounds__(VC_RESTRICT_THREADS) k_vc_restrict(int nc, const int* __restrict__ rptr,
                                                                     const int* __restrict__ rcol,
                                                                     const T* __restrict__ rv, const T* __restrict__ rf,
                                                                     const T* __restrict__ dinvc, T* __restrict__ rc,
                                                                     T* __restrict__ dc, const T* __restrict__ coefc,
                                                                     int nfine) {
  __shared__ T sh[4][AMG_NS];
  const int a = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T s[AMG_NS];
  vc_restrict_part<T, BF>(a, threadIdx.x, s, rptr, rcol, rv, rf, nfine);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < AMG_NS; q++) sh[w][q] = s[q];
  __syncthreads();
  if (threadIdx.x == 0) vc_restrict_finish<T>(a, sh, dinvc, rc, dc, coefc);
}

// coarsest solve: x = inv b (one block)
template <class T>
__global__ void k_vc_dense(int N, const T* __restrict__ inv, const T* __restrict__ b, T* __restrict__ x) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    T s = T(0);
    for (int j = 0; j < N; j++) s += inv[(int64_t)i * N + j] * b[j];
    x[i] = s;
  }
}

// prolongation: e_i = (P xc)_i, x_i += e_i.  LPR lanes per fine row: a P row
// holds the few aggregates around the node (about 7 at level 0), so a whole
// warp per row would idle most lanes (4 lanes: two blocks each, in flight
// together); P is tiled, so the lanes of a warp
// (consecutive rows, consecutive blocks) read each component in one run.
// Rows of wholly absent nodes have no blocks: their e stays zero.
// thread t of the prolongation (row t / LPR, lane t % LPR); every lane of
// the warp calls it (the row sums are reduced across the row's lanes)
template <class T, int BF, int LPR>
__device__ __forceinline__ void vc_prolong_thread(int64_t t, int n, const int* pptr, const int* pcol, const T* pv,
                                                  const T* xc, T* x, T* e, int ncoarse) {
  const int i = (int)(t / LPR);
  const int l = (int)(t % LPR);
  const bool active = i < n;
  T s[BF], xo[BF];
#pragma unroll
  for (int q = 0; q < BF; q++) s[q] = xo[q] = T(0);
  if (active && l == 0)  // the row's x, loaded ahead of its products
#pragma unroll
    for (int q = 0; q < BF; q++) xo[q] = x[(int64_t)BF * i + q];
  if (active)
    for (int k = pptr[i] + l; k < pptr[i + 1]; k += LPR) {
      const int a = fe_idx(__ldg(pcol + k), ncoarse);
      T c[AMG_NS];
#pragma unroll
      for (int j = 0; j < AMG_NS; j++) c[j] = xc[(int64_t)AMG_NS * a + j];
#pragma unroll
      for (int q = 0; q < BF; q++)
#pragma unroll
        for (int j = 0; j < AMG_NS; j++) s[q] += __ldg(pv + tix<BF * AMG_NS>(k, AMG_NS * q + j)) * c[j];
    }
#pragma unroll
  for (int q = 0; q < BF; q++)
    for (int off = LPR / 2; off > 0; off >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off, LPR);
  if (!active || l != 0) return;
#pragma unroll
  for (int q = 0; q < BF; q++) {
    e[(int64_t)BF * i + q] = s[q];
    x[(int64_t)BF * i + q] = xo[q] + s[q];
  }
}

template <class T, int BF, int LPR>
__global__ void __launch_bounds__(256) k_vc_prolong(int n, const int* __restrict__ pptr, const int* __restrict__ pcol,
                                                    const T* __restrict__ pv, const T* __restrict__ xc,
                                                    T* __restrict__ x, T* __restrict__ e, int ncoarse) {
  vc_prolong_thread<T, BF, LPR>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, n, pptr, pcol, pv, xc, x, e, ncoarse);
}

// The bottom of the V-cycle in one block (FP32).  The smallest coarse levels'
// kernels cost their launches, not bytes: levels q0..L-1 (each at most
// VC_BOTTOM_MAXNNZ blocks, q0 >= 1) run as one launch of one block --
// smoothing, restriction, the coarsest solve, prolongation and smoothing
// again, separated by block barriers.  Each stage runs the same device
// functions as the per-level kernels, with the same assignment of rows and
// entries to warps, lanes and 128-thread groups, so the result is identical.
// One SM works through the blocks, so the form pays for few of them only.  A
// preconditioner call whose largest fused level has n blocks, fused and as
// launches: 257 blocks 54.1 and 57.0 us, 317: 292 and 298, 393: 67.9 and 69.0,
// 455: 55.2 and 57.0, 521: 54.5 and 54.4, 566: 87.4 and 86.5; V-cycles alone
// with 884: 72 and 71 us, 1,794: 80 and 68, 4,267: 122 and 69, 9,073: 195 and
// 86.  The gain is 2 to 5% up to about 500 blocks and none to the line.  In FP64
// (884: 208 and 133 us; 317: 1,022 and 983) the launches win throughout.
constexpr int VC_BOTTOM_THREADS = 1024;
constexpr int64_t VC_BOTTOM_MAXNNZ = 640;

template <class T>
struct VcLevelArgs {  // one level of the bottom (device pointers)
  int n, nc;
  const int *ptr, *col;            // A_l pattern, tiled values, block-Jacobi inverse, Chebyshev coefficients
  const T *val, *dinv, *coef;
  const int *rptr, *rcol;          // P_l^T (l below the coarsest)
  const T* rv;
  const int *pptr, *pcol;          // P_l, tiled
  const T* pv;
  const T* inv;                    // coarsest: dense inverse
  T *x, *r, *d0, *d1, *e;          // V-cycle vectors
};
template <class T>
struct VcBottomArgs {
  int nb;                          // levels q0 .. q0 + nb - 1, the last one the coarsest
  VcLevelArgs<T> lev[AMG_MAXLEV];
};

template <class T>
__global__ void __launch_bounds__(VC_BOTTOM_THREADS) k_vc_bottom(const VcBottomArgs<T> P) {
  constexpr int NT = VC_BOTTOM_THREADS;
  constexpr int NW = NT / 32;
  constexpr int NG = NT / VC_RESTRICT_THREADS;
  __shared__ T sh[NG][4][AMG_NS];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // one Chebyshev step of a level: rows strided over the warps
  auto cheb = [&](const VcLevelArgs<T>& L, const T* g, T* dout, T cx, int flags) {
    for (int row = wid; row < L.n; row += NW)
      vc_cheb_row<T, AMG_NS>(row, lane, L.n, L.ptr, L.col, L.val, L.dinv, g, L.x, L.r, dout, cx, L.coef, flags);
    __syncthreads();
  };
  const int nb = P.nb;
  for (int l = 0; l < nb - 1; l++) {  // downward
    const VcLevelArgs<T>& L = P.lev[l];
    const VcLevelArgs<T>& C = P.lev[l + 1];
    cheb(L, L.d0, L.d1, T(1), VC_SETX);
    cheb(L, L.d1, nullptr, T(1), 0);
    const bool coarsest = l + 1 == nb - 1;
    const int grp = tid / VC_RESTRICT_THREADS, t = tid % VC_RESTRICT_THREADS, w = t >> 5;
    for (int a0 = 0; a0 < C.n; a0 += NG) {  // coarse rows, one per 128-thread group
      const int a = a0 + grp;
      if (a < C.n) {
        T s[AMG_NS];
        vc_restrict_part<T, AMG_NS>(a, t, s, L.rptr, L.rcol, L.rv, L.r, L.n);
        if (lane == 0)
#pragma unroll
          for (int q = 0; q < AMG_NS; q++) sh[grp][w][q] = s[q];
      }
      __syncthreads();
      if (t == 0 && a < C.n) vc_restrict_finish<T>(a, sh[grp], C.dinv, C.r, coarsest ? nullptr : C.d0, C.coef);
      __syncthreads();
    }
  }
  {  // coarsest: x = inv r
    const VcLevelArgs<T>& Lc = P.lev[nb - 1];
    const int N = Lc.n * AMG_NS;
    for (int i = tid; i < N; i += NT) {
      T s = T(0);
      for (int j = 0; j < N; j++) s += Lc.inv[(int64_t)i * N + j] * Lc.r[j];
      Lc.x[i] = s;
    }
    __syncthreads();
  }
  for (int l = nb - 2; l >= 0; l--) {  // upward
    const VcLevelArgs<T>& L = P.lev[l];
    const VcLevelArgs<T>& C = P.lev[l + 1];
    constexpr int LPR = 4;
    for (int64_t t0 = 0; t0 < (int64_t)L.n * LPR; t0 += NT)
      vc_prolong_thread<T, AMG_NS, LPR>(t0 + tid, L.n, L.pptr, L.pcol, L.pv, C.x, L.x, L.e, L.nc);
    __syncthreads();
    cheb(L, L.e, L.d0, T(0), VC_KEEPX | VC_START);
    cheb(L, L.d0, L.d1, T(1), VC_FINAL);
  }
}

template <class A, class B>
__global__ void k_vc_convert(int64_t n, const A* __restrict__ a, B* __restrict__ b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (B)a[i];
}
// ---------------------------------------------------------------- host drivers
template <class X>
int dev_alloc(fe_mesh m, X** p, size_t count) {
  count = count ? count : 1;
  FE_TRY(fe_alloc_t(m, p, count));
  m->amg->allocs.push_back((void*)*p);
  m->amg->bytes += (int64_t)(count * sizeof(X));
  return FE_OK;
}

// an array the hierarchy can do without: *p stays null where it does not fit
template <class X>
int dev_alloc_optional(fe_mesh m, X** p, size_t count) {
  if (m->lean) return FE_OK;
  const int rc = fe_alloc_once(m, reinterpret_cast<void**>(p), std::max<size_t>(count, 1) * sizeof(X));
  if (rc == FE_ERR_OOM) return FE_OK;
  FE_TRY(rc);
  m->amg->allocs.push_back((void*)*p);
  m->amg->bytes += (int64_t)(std::max<size_t>(count, 1) * sizeof(X));
  return FE_OK;
}

template <class X>
int upload(fe_mesh m, X** p, const std::vector<X>& v) {
  FE_TRY(dev_alloc(m, p, v.size()));
  if (!v.empty()) FE_CUDA(cudaMemcpyAsync(*p, v.data(), v.size() * sizeof(X), cudaMemcpyHostToDevice, m->stream));
  return FE_OK;
}

unsigned blocks_for(int64_t n, int per) { return (unsigned)std::max<int64_t>(1, (n + per - 1) / per); }

// structure of every level, once per mesh
int build_structure(fe_mesh m) {
  AmgHier* h = m->amg;
  std::vector<HostLevel> hl(1);
  HostLevel& L0 = hl[0];
  const int nn = m->nn;
  L0.n = nn;
  L0.b = 3;
  L0.ptr.resize(nn + 1);
  L0.col.resize(m->nnzb);
  std::vector<uint8_t> fix(nn);
  std::vector<double> X((size_t)nn * 3);
  FE_CUDA(cudaMemcpyAsync(L0.ptr.data(), m->row_ptr, sizeof(int) * (nn + 1), cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaMemcpyAsync(L0.col.data(), m->col, sizeof(int) * m->nnzb, cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaMemcpyAsync(fix.data(), m->fixmask, nn, cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaMemcpyAsync(X.data(), m->X, sizeof(double) * 3 * nn, cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  L0.absent = fix;
  L0.ns.assign((size_t)nn * 3 * AMG_NS, 0.0);
  for (int a = 0; a < nn; a++) {
    const double x = X[3 * a], y = X[3 * a + 1], z = X[3 * a + 2];
    const double rb[3][AMG_NS] = {{1, 0, 0, -y, 0, z}, {0, 1, 0, x, -z, 0}, {0, 0, 1, 0, y, -x}};
    for (int c = 0; c < 3; c++)
      for (int k = 0; k < AMG_NS; k++) L0.ns[((size_t)3 * a + c) * AMG_NS + k] = ((fix[a] >> c) & 1) ? 0.0 : rb[c][k];
  }
  int l = 0;
  for (;;) {
    HostLevel& L = hl[l];
    if (L.n <= AMG_COARSE || l == AMG_MAXLEV - 1) break;
    aggregate(L);
    if (L.nc == 0 || L.nc > 0.9 * L.n) {
      L.agg.clear();
      L.nc = 0;
      break;
    }
    hl.emplace_back();
    coarsen(hl[l], hl[l + 1]);
    l++;
  }
  const int nlev = l + 1;
  const HostLevel& Lc = hl[nlev - 1];
  if (Lc.n * Lc.b > AMG_DENSE_MAX)
    return fe_set_error("AMG: the coarsest level has %d unknowns (at most %d)", Lc.n * Lc.b, AMG_DENSE_MAX),
           FE_ERR_ARG;
  h->nlev = nlev;
  for (int q = 0; q < nlev; q++) {
    HostLevel& H = hl[q];
    AmgLevel& A = h->lev[q];
    A.n = H.n;
    A.b = H.b;
    A.nc = q < nlev - 1 ? H.nc : 0;
    if (q == 0) {
      A.ptr = m->row_ptr;
      A.col = m->col;
      A.diag = m->diag_pos;
      A.nnz = m->nnzb;
    } else {
      int *p = nullptr, *c = nullptr, *d = nullptr;
      FE_TRY(upload(m, &p, H.ptr));
      FE_TRY(upload(m, &c, H.col));
      FE_TRY(upload(m, &d, H.diag));
      A.ptr = p;
      A.col = c;
      A.diag = d;
      A.nnz = (int64_t)H.col.size();
    }
    FE_TRY(upload(m, &A.absent, H.absent));
    if (q < nlev - 1) {
      FE_TRY(upload(m, &A.agg, H.agg));
      FE_TRY(upload(m, &A.pptr, H.pptr));
      FE_TRY(upload(m, &A.pcol, H.pcol));
      std::vector<int> prow(H.pcol.size());
      for (int i = 0; i < H.n; i++)
        for (int k = H.pptr[i]; k < H.pptr[i + 1]; k++) prow[k] = i;
      FE_TRY(upload(m, &A.prow, prow));
      FE_TRY(upload(m, &A.rptr, H.rptr));
      FE_TRY(upload(m, &A.rcol, H.rcol));
      FE_TRY(upload(m, &A.rsrc, H.rsrc));
      FE_TRY(upload(m, &A.apptr, H.apptr));
      FE_TRY(upload(m, &A.apcol, H.apcol));
      FE_TRY(upload(m, &A.tnode, H.tnode));
      A.nnzp = (int64_t)H.pcol.size();
      A.nnzr = A.nnzp;
      A.nnzap = (int64_t)H.apcol.size();
      FE_TRY(dev_alloc(m, &A.pk_ptr, (size_t)A.nnzp));
      FE_TRY(dev_alloc(m, &A.pk, (size_t)A.nnz));
      FE_TRY(dev_alloc(m, &A.rpos, (size_t)A.nnzr));
      k_amg_plists<<<blocks_for(A.n, 128), 128, 0, m->stream>>>(A.n, A.ptr, A.col, A.agg, A.pptr, A.pcol, A.pk_ptr,
                                                                A.pk);
      k_amg_rpos<<<blocks_for(A.nnzr, 256), 256, 0, m->stream>>>(A.nnzr, A.rsrc, A.rpos);
      FE_CUDA(cudaGetLastError());
      FE_TRY(upload(m, &A.apoff, H.apoff));
      FE_TRY(upload(m, &A.raoff, H.raoff));
      A.napidx = H.apoff.back();
      A.nralist = H.raoff.back();
      FE_TRY(dev_alloc(m, &A.tnode32, H.tnode.size()));
      k_amg_to_f32<<<blocks_for((int64_t)H.tnode.size(), 256), 256, 0, m->stream>>>((int64_t)H.tnode.size(), A.tnode,
                                                                                   A.tnode32);
      FE_CUDA(cudaGetLastError());
    }
  }
  for (int q = 0; q < nlev - 1; q++) {
    AmgLevel &A = h->lev[q], &Cq = h->lev[q + 1];
    FE_TRY(dev_alloc(m, &A.lend, (size_t)Cq.nnz));
    FE_TRY(dev_alloc(m, &A.crow, (size_t)Cq.nnz));
    FE_TRY(dev_alloc_optional(m, &A.apidx, (size_t)A.napidx));
    FE_TRY(dev_alloc_optional(m, &A.ralist, (size_t)A.nralist));
    if (A.apidx)
      k_amg_apidx<<<blocks_for((int64_t)A.n * 32, 256), 256, 0, m->stream>>>(A.n, A.ptr, A.col, A.pptr, A.pcol, A.apptr,
                                                                           A.apcol, A.apoff, A.apidx);
    k_amg_raplists<<<blocks_for((int64_t)Cq.n * 32, 256), 256, 0, m->stream>>>(
        Cq.n, Cq.ptr, Cq.col, A.rptr, A.rcol, A.rsrc, A.apptr, A.apcol, A.raoff, A.lend, A.crow, A.ralist);
    FE_CUDA(cudaGetLastError());
  }
  int64_t maxN = 0;
  for (int q = 0; q < nlev; q++) maxN = std::max<int64_t>(maxN, (int64_t)h->lev[q].n * h->lev[q].b);
  FE_TRY(dev_alloc(m, &h->pw, (size_t)2 * maxN));
  const size_t blocks = std::max<size_t>(stream_grid(m->warps64), (size_t)POWER_BLOCKS_PER_SM * m->sm_count);
  FE_TRY(dev_alloc(m, &h->part, 2 * blocks));
  FE_TRY(dev_alloc(m, &h->ticket, 4));
  FE_CUDA(cudaMemsetAsync(h->ticket, 0, 4 * sizeof(unsigned), m->stream));
  FE_TRY(dev_alloc(m, &h->scal, (size_t)AMG_MAXLEV * SC_N));
  FE_CUDA(cudaStreamSynchronize(m->stream));  // host vectors above go out of scope
  return FE_OK;
}

// the arrays of the setup's arithmetic type C
template <class C>
struct Arr {
  static C*& val(AmgLevel& L);
  static C*& dinv(AmgLevel& L);
  static C*& p(AmgLevel& L);
  static C*& ap(AmgLevel& L);
  static C*& r(AmgLevel& L);
  static C*& pt(AmgLevel& L);
};
template <>
struct Arr<double> {
  static double*& val(AmgLevel& L) { return L.val64; }
  static double*& dinv(AmgLevel& L) { return L.dinv64; }
  static double*& p(AmgLevel& L) { return L.p64; }
  static double*& ap(AmgLevel& L) { return L.ap64; }
  static double*& r(AmgLevel& L) { return L.r64; }
  static double*& pt(AmgLevel& L) { return L.pt64; }
};
template <>
struct Arr<float> {
  static float*& val(AmgLevel& L) { return L.val32; }
  static float*& dinv(AmgLevel& L) { return L.dinv32; }
  static float*& p(AmgLevel& L) { return L.p32; }
  static float*& ap(AmgLevel& L) { return L.ap32; }
  static float*& r(AmgLevel& L) { return L.r32; }
  static float*& pt(AmgLevel& L) { return L.pt32; }
};

// one power step of level q, x -> y
template <class C, class V, int B>
int power_step(fe_mesh m, AmgLevel& L, const V* A, const C* dinv, const C* x, C* y, const PowerArgs& pa, bool last) {
  FE_SCOPE(m, FE_PROF_OTHER, (double)L.nnz * (B * B * sizeof(V) + 4) + 2.0 * sizeof(C) * L.n * B);
  if constexpr (B == 3 && sizeof(C) == 8)
    k_amg_power0<C, V><<<stream_grid(m->warps64), STREAM_THREADS, 0, m->stream>>>(
        L.n, m->warps64, m->ranges64, m->part64, L.ptr, L.col, A, dinv, x, y, pa, last);
  else
    k_amg_power<C, V, B><<<std::min<unsigned>(blocks_for((int64_t)L.n * 32, 256), POWER_BLOCKS_PER_SM * m->sm_count),
                           256, 0, m->stream>>>(L.n, L.ptr, L.col, Vals<C, V, B>{A}, dinv, x, y, pa, last);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// numbers of level q (A_q already numeric) in arithmetic type C: D^-1, rho,
// P (with its tiled copy and transpose), AP and A_{q+1}; the coarsest level's
// dense inverse (FP64, with an FP32 copy for the mixed forms).  Everything is
// queued; the host reads nothing.
template <class C, class V, int B>
int numeric_level(fe_mesh m, int q, const V* val) {
  AmgHier* h = m->amg;
  AmgLevel& L = h->lev[q];
  const Vals<C, V, B> A{val};
  const int64_t N = (int64_t)L.n * L.b;
  C*& dinv = Arr<C>::dinv(L);
  if (!dinv) FE_TRY(dev_alloc(m, &dinv, (size_t)L.n * B * B));
  {
    FE_SCOPE(m, FE_PROF_OTHER, (double)L.n * B * B * (8 + sizeof(C)));
    if constexpr (B == 3)
      k_amg_dinv3<C, V><<<blocks_for(L.n, 128), 128, 0, m->stream>>>(L.n, L.diag, A, dinv);
    else
      k_amg_dinv6<C, V><<<blocks_for((int64_t)L.n * 16, 128), 128, 0, m->stream>>>(L.n, L.diag, A, dinv);
  }
  FE_CUDA(cudaGetLastError());
  if (q == h->nlev - 1) {  // coarsest: dense inverse
    const int Nd = L.n * B;
    if (!L.inv64) FE_TRY(dev_alloc(m, &L.inv64, (size_t)Nd * Nd));
    if (sizeof(C) == 4 && !L.inv32) FE_TRY(dev_alloc(m, &L.inv32, (size_t)Nd * Nd));
    const int smem = (Nd * Nd + 2 * Nd) * (int)sizeof(double);
    FE_TRY(fe_kernel_smem((const void*)k_amg_dense_inverse<C, V, B>, smem));
    FE_SCOPE(m, FE_PROF_OTHER, 8.0 * Nd * Nd);
    k_amg_dense_inverse<C, V, B><<<1, 1024, smem, m->stream>>>(L.n, L.ptr, L.col, A, L.inv64,
                                                              sizeof(C) == 4 ? L.inv32 : nullptr);
    FE_CUDA(cudaGetLastError());
    return FE_OK;
  }
  // rho: power steps on D^-1 A
  if (!L.coef64) FE_TRY(dev_alloc(m, &L.coef64, 4));
  if (!L.coef32) FE_TRY(dev_alloc(m, &L.coef32, 4));
  double* scal = h->scal + q * SC_N;
  const PowerArgs pa{h->part, h->ticket, scal, L.coef64, L.coef32};
  C* x = (C*)h->pw;
  C* y = x + N;
  k_amg_start<C><<<blocks_for(N, 256), 256, 0, m->stream>>>(N, x, scal);
  FE_CUDA(cudaGetLastError());
  bool small = false;
  if constexpr (B == AMG_NS && sizeof(C) == 4) {
    if (L.nnz <= AMG_POWER_SMALL) {
      small = true;
      FE_SCOPE(m, FE_PROF_OTHER, AMG_POWER_STEPS * ((double)L.nnz * (B * B * sizeof(V) + 4) + 2.0 * sizeof(C) * N));
      k_amg_power_small<<<1, 512, 0, m->stream>>>(L.n, AMG_POWER_STEPS, L.ptr, L.col, A, dinv, x, y, pa);
      FE_CUDA(cudaGetLastError());
    }
  }
  if (!small)
    for (int it = 0; it < AMG_POWER_STEPS; it++) {
      FE_TRY((power_step<C, V, B>(m, L, val, dinv, x, y, pa, it == AMG_POWER_STEPS - 1)));
      std::swap(x, y);
    }
  C*& p = Arr<C>::p(L);
  C*& ap = Arr<C>::ap(L);
  C*& r = Arr<C>::r(L);
  C*& pt = Arr<C>::pt(L);
  if (!p) FE_TRY(dev_alloc(m, &p, (size_t)L.nnzp * B * AMG_NS));
  if (!pt) FE_TRY(dev_alloc(m, &pt, (size_t)tiled_count(L.nnzp, B * AMG_NS)));
  if (!ap) FE_TRY(dev_alloc(m, &ap, (size_t)L.nnzap * B * AMG_NS));
  if (!r) FE_TRY(dev_alloc(m, &r, (size_t)L.nnzr * B * AMG_NS));
  AmgLevel& Cq = h->lev[q + 1];
  C*& cval = Arr<C>::val(Cq);
  if (!cval) FE_TRY(dev_alloc(m, &cval, (size_t)Cq.nnz * AMG_NS * AMG_NS));
  {
    FE_SCOPE(m, FE_PROF_OTHER, 3.0 * L.nnzp * B * AMG_NS * sizeof(C));
    const C* tn = nullptr;
    if constexpr (sizeof(C) == 8) tn = L.tnode;
    else tn = L.tnode32;
    k_amg_pvals<C, V, B><<<blocks_for(L.nnzp * B, B == 3 ? 192 : 64), B == 3 ? 192 : 64, 0, m->stream>>>(
        L.nnzp, L.prow, L.pcol, L.pk_ptr, L.pk, L.col, A, L.agg, dinv, tn, scal, L.rpos, p, pt, r);
  }
  FE_CUDA(cudaGetLastError());
  {
    FE_SCOPE(m, FE_PROF_OTHER, (double)L.nnzap * B * AMG_NS * sizeof(C));
    constexpr int W = ap_warps<C, B>();
    const int smem = W * (int)sizeof(ApShared<C, B>);
    auto kern = L.apidx ? k_amg_ap<C, V, B, true> : k_amg_ap<C, V, B, false>;
    FE_TRY(fe_kernel_smem((const void*)kern, smem));
    kern<<<blocks_for(L.n, W), 32 * W, smem, m->stream>>>(L.n, L.ptr, L.col, A, L.pptr, L.pcol, p, L.apptr, L.apcol,
                                                          L.apoff, L.apidx, ap);
  }
  FE_CUDA(cudaGetLastError());
  {
    FE_SCOPE(m, FE_PROF_OTHER, (double)Cq.nnz * AMG_NS * AMG_NS * sizeof(C));
    auto kern = L.ralist ? k_amg_rap<C, B, true> : k_amg_rap<C, B, false>;
    kern<<<blocks_for(Cq.nnz * (B == 3 ? AMG_NS : AMG_NS * AMG_NS), B == 3 ? 192 : 64), B == 3 ? 192 : 64, 0, m->stream>>>(
        Cq.nnz, L.crow, Cq.col, L.lend, L.raoff, L.ralist, L.rptr, L.rcol, L.rsrc, L.apptr, L.apcol, p, ap, Cq.absent,
        cval);
  }
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// the whole hierarchy's numbers: FP64 for an FP64 tangent, FP32 otherwise
template <class C, class V>
int numeric_all(fe_mesh m, const V* K0) {
  AmgHier* h = m->amg;
  FE_TRY((numeric_level<C, V, 3>(m, 0, K0)));
  for (int q = 1; q < h->nlev; q++) FE_TRY((numeric_level<C, C, AMG_NS>(m, q, Arr<C>::val(h->lev[q]))));
  double sc[AMG_MAXLEV * SC_N];
  FE_CUDA(cudaMemcpyAsync(sc, h->scal, sizeof(sc), cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  for (int q = 0; q < h->nlev - 1; q++) {
    const double rho = sc[q * SC_N + SC_RHO];
    if (!(rho > 0.0) || !std::isfinite(rho))
      return fe_set_error("AMG: spectral radius estimate %g on level %d", rho, q), FE_ERR_STATE;
    h->lev[q].rho = rho;
  }
  return FE_OK;
}

int ensure_vectors(fe_mesh m, int elem) {
  AmgHier* h = m->amg;
  if (h->vec_elem == elem) return FE_OK;  // (a precision change allocates a new set)
  for (int q = 0; q < h->nlev; q++) {
    AmgLevel& L = h->lev[q];
    const size_t bytes = (size_t)L.n * L.b * elem;
    if (q == 0) L.x = m->zx;  // allocated before any preconditioner application
    void** vs[5] = {&L.r, &L.d0, &L.d1, &L.e, &L.x};
    for (void** v : vs) {
      if (q == 0 && v == &L.x) continue;
      char* p = nullptr;
      FE_TRY(dev_alloc(m, &p, bytes));
      *v = p;
    }
  }
  h->vec_elem = elem;
  return FE_OK;
}

// The kernels of one V-cycle in precision T, level-0 values of type V
// (tiled), on stream st: input b (FP64 [3 nn], read by the first kernel
// alone), result in lev[0].x.  Adds the algorithmic bytes and flops of its
// kernels to *bytes, *flops.
template <class T, class V>
int vcycle_launches(fe_mesh m, cudaStream_t st, const V* K0, const double* b, double* bytes, double* flops) {
  AmgHier* h = m->amg;
  const int L = h->nlev;
  constexpr bool D = sizeof(T) == 8;
  auto vals = [&](int q) -> const T* { return D ? (const T*)h->lev[q].val64 : (const T*)h->lev[q].val32; };
  auto dinv = [&](int q) -> const T* { return D ? (const T*)h->lev[q].dinv64 : (const T*)h->lev[q].dinv32; };
  auto pv = [&](int q) -> const T* { return D ? (const T*)h->lev[q].pt64 : (const T*)h->lev[q].pt32; };
  auto rv = [&](int q) -> const T* { return D ? (const T*)h->lev[q].r64 : (const T*)h->lev[q].r32; };
  auto inv = [&](int q) -> const T* { return D ? (const T*)h->lev[q].inv64 : (const T*)h->lev[q].inv32; };
  auto coef = [&](int q) -> const T* { return D ? (const T*)h->lev[q].coef64 : (const T*)h->lev[q].coef32; };
  auto X = [&](int q) { return (T*)h->lev[q].x; };
  const double sv = sizeof(T), s0 = sizeof(V);
  // level 0: the scan form where its 16-row groups fill the wave four times
  // (FP32 and BF16 values; see k_vc_cheb0_scan)
  unsigned grid_scan = 0;
  if constexpr (!D) {
    int per_sm = 0;
    FE_TRY(fe_kernel_occupancy((const void*)k_vc_cheb0_scan<V, T>, 256, 0, &per_sm));
    const int64_t groups = ((int64_t)m->nn + VC_RPW - 1) / VC_RPW, wave = (int64_t)std::max(per_sm, 1) * m->sm_count;
    if (groups >= 4 * 8 * wave) grid_scan = (unsigned)wave;
  }
  // Chebyshev step on level q (fused SpMV)
  auto step = [&](int q, const T* g, T* dout, double cx, int flags) -> int {
    AmgLevel& Lq = h->lev[q];
    const int B = Lq.b;
    *bytes += (double)Lq.nnz * (B * B * (q == 0 ? s0 : sv) + 4) + 4.0 * (Lq.n + 1) + (double)Lq.n * B * (sv * 5 + B * sv);
    *flops += 2.0 * Lq.nnz * B * B;
    if constexpr (!D)
      if (q == 0 && grid_scan) {
        k_vc_cheb0_scan<V, T><<<grid_scan, 256, 0, st>>>(Lq.n, Lq.ptr, Lq.col, K0, dinv(0), g, X(0), (T*)Lq.r, dout,
                                                         (T)cx, coef(0), flags);
        FE_CUDA(cudaGetLastError());
        return FE_OK;
      }
    if (q == 0)
      k_vc_cheb0<V, T><<<stream_grid(h->shape0.warps), STREAM_THREADS, 0, st>>>(
          Lq.n, h->shape0.warps, h->shape0.ranges, h->part0, Lq.ptr, Lq.col, K0, dinv(0), g, X(0), (T*)Lq.r, dout,
          (T)cx, coef(0), flags);
    else
      k_vc_cheb<T, AMG_NS><<<blocks_for((int64_t)Lq.n * 32, VC_CHEB_THREADS<T>), VC_CHEB_THREADS<T>, 0, st>>>(
          Lq.n, Lq.ptr, Lq.col, vals(q), dinv(q), g, X(q), (T*)Lq.r, dout, (T)cx, coef(q), flags);
    FE_CUDA(cudaGetLastError());
    return FE_OK;
  };
  if (L == 1) {  // one level: the exact solve
    AmgLevel& L0 = h->lev[0];
    const int64_t N = (int64_t)L0.n * 3;
    k_vc_convert<double, T><<<blocks_for(N, 256), 256, 0, st>>>(N, b, (T*)L0.r);
    k_vc_dense<T><<<1, 256, 0, st>>>((int)N, inv(0), (const T*)L0.r, X(0));
    FE_CUDA(cudaGetLastError());
    *bytes += (double)N * N * sv + 8.0 * N;
    *flops += 2.0 * N * N;
    return FE_OK;
  }
  // the bottom levels q0..L-1 (at most VC_BOTTOM_MAXNNZ blocks each, q0 >= 1)
  // run in one block when at least one of them is smoothed
  int q0 = L - 1;
  while (!D && q0 > 1 && h->lev[q0 - 1].nnz <= VC_BOTTOM_MAXNNZ) q0--;
  const bool fused = q0 <= L - 2;
  const int qf = fused ? q0 : L - 1;  // the per-level kernels run on levels 0..qf-1
  // downward: pre-smoothing, restriction
  for (int q = 0; q < qf; q++) {
    AmgLevel& Lq = h->lev[q];
    if (q == 0) {
      k_vc_init0<T><<<blocks_for(Lq.n, 256), 256, 0, st>>>(Lq.n, dinv(0), b, (T*)Lq.r, (T*)Lq.d0, coef(0));
      FE_CUDA(cudaGetLastError());
      *bytes += (double)Lq.n * (24 + 9 * sv + 6 * sv);
    }
    // x = d0; r -= A d0; d1 = c1 d0 + c2 D^-1 r
    FE_TRY(step(q, (const T*)Lq.d0, (T*)Lq.d1, 1.0, VC_SETX));
    // x += d1; r -= A d1 (r = b - A x for the restriction)
    FE_TRY(step(q, (const T*)Lq.d1, nullptr, 1.0, 0));
    AmgLevel& Cq = h->lev[q + 1];
    const bool coarsest = q + 1 == L - 1;
    *bytes += (double)Lq.nnzr * (Lq.b * AMG_NS * sv + 4) + (double)Lq.n * Lq.b * sv + (double)Cq.n * AMG_NS * sv * 2;
    *flops += 2.0 * Lq.nnzr * Lq.b * AMG_NS;
    if (Lq.b == 3)
      k_vc_restrict<T, 3><<<Cq.n, 128, 0, st>>>(Cq.n, Lq.rptr, Lq.rcol, rv(q), (const T*)Lq.r, dinv(q + 1), (T*)Cq.r,
                                                coarsest ? nullptr : (T*)Cq.d0, coef(q + 1), Lq.n);
    else
      k_vc_restrict<T, AMG_NS><<<Cq.n, 128, 0, st>>>(Cq.n, Lq.rptr, Lq.rcol, rv(q), (const T*)Lq.r, dinv(q + 1),
                                                     (T*)Cq.r, coarsest ? nullptr : (T*)Cq.d0, coef(q + 1), Lq.n);
    FE_CUDA(cudaGetLastError());
  }
  if (fused) {  // levels q0..L-1 in one block (the bytes and flops of the kernels it replaces)
    VcBottomArgs<T> a{};
    a.nb = L - q0;
    for (int l = 0; l < a.nb; l++) {
      AmgLevel& Lq = h->lev[q0 + l];
      VcLevelArgs<T>& A = a.lev[l];
      A.n = Lq.n;
      A.nc = Lq.nc;
      A.ptr = Lq.ptr;
      A.col = Lq.col;
      A.val = vals(q0 + l);
      A.dinv = dinv(q0 + l);
      A.coef = coef(q0 + l);
      A.rptr = Lq.rptr;
      A.rcol = Lq.rcol;
      A.rv = rv(q0 + l);
      A.pptr = Lq.pptr;
      A.pcol = Lq.pcol;
      A.pv = pv(q0 + l);
      A.inv = l == a.nb - 1 ? inv(q0 + l) : nullptr;
      A.x = X(q0 + l);
      A.r = (T*)Lq.r;
      A.d0 = (T*)Lq.d0;
      A.d1 = (T*)Lq.d1;
      A.e = (T*)Lq.e;
      if (l < a.nb - 1) {
        const AmgLevel& Cq = h->lev[q0 + l + 1];
        const int B = Lq.b;
        *bytes += 4 * ((double)Lq.nnz * (B * B * sv + 4) + 4.0 * (Lq.n + 1) + (double)Lq.n * B * (sv * 5 + B * sv));
        *flops += 4 * 2.0 * Lq.nnz * B * B;
        *bytes += (double)Lq.nnzr * (B * AMG_NS * sv + 4) + (double)Lq.n * B * sv + (double)Cq.n * AMG_NS * sv * 2;
        *flops += 2.0 * Lq.nnzr * B * AMG_NS;
        *bytes += (double)Lq.nnzp * (B * AMG_NS * sv + 4) + (double)Lq.n * B * sv * 3;
        *flops += 2.0 * Lq.nnzp * B * AMG_NS;
      } else {
        const int N = Lq.n * Lq.b;
        *bytes += (double)N * N * sv;
        *flops += 2.0 * N * N;
      }
    }
    if constexpr (!D) k_vc_bottom<T><<<1, VC_BOTTOM_THREADS, 0, st>>>(a);
    FE_CUDA(cudaGetLastError());
  } else {  // coarsest
    AmgLevel& Lc = h->lev[L - 1];
    const int N = Lc.n * Lc.b;
    k_vc_dense<T><<<1, 256, 0, st>>>(N, inv(L - 1), (const T*)Lc.r, X(L - 1));
    FE_CUDA(cudaGetLastError());
    *bytes += (double)N * N * sv;
    *flops += 2.0 * N * N;
  }
  // upward: prolongation, post-smoothing
  for (int q = qf - 1; q >= 0; q--) {
    AmgLevel& Lq = h->lev[q];
    *bytes += (double)Lq.nnzp * (Lq.b * AMG_NS * sv + 4) + (double)Lq.n * Lq.b * sv * 3;
    *flops += 2.0 * Lq.nnzp * Lq.b * AMG_NS;
    const unsigned grid = blocks_for((int64_t)Lq.n * 4, 256);
    if (Lq.b == 3)
      k_vc_prolong<T, 3, 4><<<grid, 256, 0, st>>>(Lq.n, Lq.pptr, Lq.pcol, pv(q), X(q + 1), X(q), (T*)Lq.e, Lq.nc);
    else
      k_vc_prolong<T, AMG_NS, 4><<<grid, 256, 0, st>>>(Lq.n, Lq.pptr, Lq.pcol, pv(q), X(q + 1), X(q), (T*)Lq.e,
                                                       Lq.nc);
    FE_CUDA(cudaGetLastError());
    // r -= A e; d0 = D^-1 r / theta
    FE_TRY(step(q, (const T*)Lq.e, (T*)Lq.d0, 0.0, VC_KEEPX | VC_START));
    // x += d0; r -= A d0; d1 = c1 d0 + c2 D^-1 r; x += d1
    FE_TRY(step(q, (const T*)Lq.d0, (T*)Lq.d1, 1.0, VC_FINAL));
  }
  return FE_OK;
}

void drop_graph(AmgHier* h) {
  if (h->exec) cudaGraphExecDestroy(h->exec);
  if (h->graph) cudaGraphDestroy(h->graph);
  h->exec = nullptr;
  h->graph = nullptr;
  h->root = nullptr;
}

// The captured graph's first kernel (k_vc_init0 or, with one level,
// k_vc_convert) and the place of the input vector among its arguments.
int find_root(AmgHier* h) {
  size_t n = 1;
  if (cudaGraphGetRootNodes(h->graph, &h->root, &n) != cudaSuccess || n != 1)
    return fe_set_error("the V-cycle graph has no single first kernel"), FE_ERR_CUDA;
  h->root_arg = h->nlev == 1 ? 1 : 2;
  return FE_OK;
}

// lets the graph's next launches read b
int set_input(AmgHier* h, const double* b) {
  cudaKernelNodeParams p{};
  FE_CUDA(cudaGraphKernelNodeGetParams(h->root, &p));
  void* args[8];
  for (int i = 0; i < (h->nlev == 1 ? 3 : 6); i++) args[i] = p.kernelParams[i];
  args[h->root_arg] = (void*)&b;
  p.kernelParams = args;
  FE_CUDA(cudaGraphExecKernelNodeSetParams(h->exec, h->root, &p));
  return FE_OK;
}

// capture the V-cycle of the current precision into a CUDA graph
template <class T, class V>
int capture(fe_mesh m, const V* K0, const double* b) {
  AmgHier* h = m->amg;
  drop_graph(h);
  if (!h->cap) FE_CUDA(cudaStreamCreateWithFlags(&h->cap, cudaStreamNonBlocking));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  h->shape0 = stream_shape(cheb0_blocks_per_sm<T>(), m->sm_count, m->nnzb);
  if (h->part0_len < h->shape0.ranges + 1) {
    FE_TRY(dev_alloc(m, &h->part0, (size_t)h->shape0.ranges + 1));
    h->part0_len = h->shape0.ranges + 1;
  }
  FE_TRY(fe_stream_partition(m, h->shape0.ranges, h->part0));
  double bytes = 0.0, flops = 0.0;
  m->prof_suspend++;
  cudaGraph_t g = nullptr;
  cudaError_t e0 = cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal);
  int rc = e0 == cudaSuccess ? vcycle_launches<T, V>(m, h->cap, K0, b, &bytes, &flops) : FE_ERR_CUDA;
  cudaError_t e1 = e0 == cudaSuccess ? cudaStreamEndCapture(h->cap, &g) : e0;
  m->prof_suspend--;
  if (rc != FE_OK) {
    if (g) cudaGraphDestroy(g);
    return rc;
  }
  if (e1 != cudaSuccess)
    return fe_set_error("capturing the V-cycle failed: %s", cudaGetErrorString(e1)), FE_ERR_CUDA;
  h->graph = g;
  cudaError_t e2 = cudaGraphInstantiate(&h->exec, g, 0);
  if (e2 != cudaSuccess) {
    h->exec = nullptr;
    drop_graph(h);
    return fe_set_error("instantiating the V-cycle graph failed: %s", cudaGetErrorString(e2)), FE_ERR_CUDA;
  }
  FE_TRY(find_root(h));
  h->exec_prec = m->prec;
  h->vc_bytes = bytes;
  h->vc_flops = flops;
  return FE_OK;
}

}  // namespace

int fe_amg_setup(fe_mesh m) {
  if (!m->amg) {
    m->amg = new AmgHier();
    int rc = build_structure(m);
    if (rc != FE_OK) {
      fe_amg_free(m);
      return rc;
    }
  }
  m->amg->ready = false;
  if (m->prec == FE_PREC_FP64) FE_TRY((numeric_all<double, double>(m, m->K64)));
  else if (m->prec == FE_PREC_MIXED_BF16) FE_TRY((numeric_all<float, __nv_bfloat16>(m, m->K16)));
  else FE_TRY((numeric_all<float, float>(m, m->K32)));
  m->amg->ready = true;
  m->amg->prec = m->prec;
  return FE_OK;
}

int fe_amg_apply(fe_mesh m, const double* x, double* z) {
  if (!m->amg || !m->amg->ready) return fe_set_error("AMG hierarchy not set up"), FE_ERR_STATE;
  AmgHier* h = m->amg;
  const bool d64 = m->prec == FE_PREC_FP64;
  FE_TRY(ensure_vectors(m, d64 ? 8 : 4));
  // pc_type 2 with the FP32 tangent: the smoother reads a BF16 copy of the
  // fine level (half the bytes of the V-cycle's dominant passes); coarse
  // levels, transfers and vectors stay FP32
  const bool bf_smooth = m->pc_type == 2 && m->prec == FE_PREC_MIXED_FP32;
  const int variant = bf_smooth ? 16 : m->prec;
  if (!h->exec || h->exec_prec != variant) {
    if (d64) FE_TRY((capture<double, double>(m, m->K64, x)));
    else if (m->prec == FE_PREC_MIXED_BF16 || bf_smooth) FE_TRY((capture<float, __nv_bfloat16>(m, m->K16, x)));
    else FE_TRY((capture<float, float>(m, m->K32, x)));
    h->exec_prec = variant;
  }
  FE_TRY(set_input(h, x));
  {
    FE_SCOPE_F(m, FE_PROF_PC, h->vc_bytes, h->vc_flops);
    FE_CUDA(cudaGraphLaunch(h->exec, m->stream));
  }
  if (z) {
    const int64_t N = (int64_t)m->nn * 3;
    if (d64) FE_CUDA(cudaMemcpyAsync(z, m->zx, N * sizeof(double), cudaMemcpyDeviceToDevice, m->stream));
    else k_vc_convert<float, double><<<blocks_for(N, 256), 256, 0, m->stream>>>(N, (const float*)m->zx, z);
    FE_CUDA(cudaGetLastError());
  }
  return FE_OK;
}

// Gives the product lists back (Cook P2 48x48x8: 175 MB, a fifth of what a mesh
// with the hierarchy holds); the products are searched from then on.  false:
// there were none.
bool fe_amg_release_lists(fe_mesh m) {
  AmgHier* h = m->amg;
  if (!h) return false;
  int64_t freed = 0;
  auto drop = [&](auto*& p, int64_t count) {
    if (!p) return;
    h->allocs.erase(std::find(h->allocs.begin(), h->allocs.end(), (void*)p));
    cudaFreeAsync(p, m->stream);
    freed += std::max<int64_t>(count, 1) * (int64_t)sizeof(*p);
    p = nullptr;
  };
  for (int q = 0; q < h->nlev; q++) {
    drop(h->lev[q].apidx, h->lev[q].napidx);
    drop(h->lev[q].ralist, h->lev[q].nralist);
  }
  h->bytes -= freed;
  m->device_bytes -= freed;
  return freed > 0;
}

void fe_amg_free(fe_mesh m) {
  if (!m->amg) return;
  drop_graph(m->amg);
  if (m->amg->cap) cudaStreamDestroy(m->amg->cap);
  for (void* p : m->amg->allocs) cudaFreeAsync(p, m->stream);
  m->device_bytes -= m->amg->bytes;
  delete m->amg;
  m->amg = nullptr;
}

// Copy of level `level` of the hierarchy to host buffers (each may be NULL):
// info [5] = n, b, nnz(A_l), nc, nnz(P_l); rho; A_l pattern and FP64 values
// (level 0: the tangent's own pattern and values are not copied), absent
// components, aggregates, and P_l's pattern and FP64 values.
extern "C" int fe_amg_get_level(fe_mesh m, int level, int64_t* info, double* rho, int32_t* ptr, int32_t* col,
                                double* val, uint8_t* absent, int32_t* agg, int32_t* pptr, int32_t* pcol,
                                double* pval) {
  if (!m) return fe_set_error("NULL mesh"), FE_ERR_ARG;
  if (!m->amg || !m->amg->ready) return fe_set_error("no AMG hierarchy"), FE_ERR_STATE;
  AmgHier* h = m->amg;
  if (level < 0 || level >= h->nlev) return fe_set_error("level %d outside [0, %d)", level, h->nlev), FE_ERR_ARG;
  FE_CUDA(cudaSetDevice(m->device));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  const AmgLevel& L = h->lev[level];
  const bool last = level == h->nlev - 1;
  if (info) {
    info[0] = L.n;
    info[1] = L.b;
    info[2] = L.nnz;
    info[3] = last ? 0 : L.nc;
    info[4] = last ? 0 : L.nnzp;
  }
  if (rho) *rho = L.rho;
  // values in FP64 (widened from the FP32 numbers of the mixed forms), those of
  // the last setup: the arrays of another precision may be there, too
  const bool f64 = h->prec == FE_PREC_FP64;
  auto copy_vals = [&](double* dst, const double* s64, const float* s32, int64_t count) -> int {
    if (f64) {
      FE_CUDA(cudaMemcpy(dst, s64, sizeof(double) * count, cudaMemcpyDeviceToHost));
    } else {
      std::vector<float> tmp(count);
      FE_CUDA(cudaMemcpy(tmp.data(), s32, sizeof(float) * count, cudaMemcpyDeviceToHost));
      for (int64_t i = 0; i < count; i++) dst[i] = (double)tmp[i];
    }
    return FE_OK;
  };
  if (level > 0) {
    if (ptr) FE_CUDA(cudaMemcpy(ptr, L.ptr, sizeof(int) * (L.n + 1), cudaMemcpyDeviceToHost));
    if (col) FE_CUDA(cudaMemcpy(col, L.col, sizeof(int) * L.nnz, cudaMemcpyDeviceToHost));
    if (val) FE_TRY(copy_vals(val, L.val64, L.val32, L.nnz * L.b * L.b));
  }
  if (absent) FE_CUDA(cudaMemcpy(absent, L.absent, L.n, cudaMemcpyDeviceToHost));
  if (!last) {
    if (agg) FE_CUDA(cudaMemcpy(agg, L.agg, sizeof(int) * L.n, cudaMemcpyDeviceToHost));
    if (pptr) FE_CUDA(cudaMemcpy(pptr, L.pptr, sizeof(int) * (L.n + 1), cudaMemcpyDeviceToHost));
    if (pcol) FE_CUDA(cudaMemcpy(pcol, L.pcol, sizeof(int) * L.nnzp, cudaMemcpyDeviceToHost));
    if (pval) FE_TRY(copy_vals(pval, L.p64, L.p32, L.nnzp * L.b * AMG_NS));
  }
  return FE_OK;
}

extern "C" int fe_amg_levels(fe_mesh m) { return (m && m->amg && m->amg->ready) ? m->amg->nlev : 0; }

FE_DBG_BOUNDS_READER(fe_dbg_bounds_amg)
