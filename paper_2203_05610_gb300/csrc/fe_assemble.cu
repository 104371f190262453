// fe_assemble.cu -- residual, energy and consistent-tangent assembly on
// P1/P2 tetrahedra (arxiv 2203.05610: residual form R(d) = f - div P(F),
// F = I + grad d, P = dPsi/dF; energy of Eq. "minimization"; tangent of
// Eq. "newton"), materials of Section "Test problems and solvers details".
//
// Residual: one thread per element (few P2 elements: per quadrature point, the
// lanes reduced with warp shuffles) writes its contributions, then one thread per
// node gathers its incident contributions in a fixed order, adds loads and
// springs, masks prescribed components and reduces ||R||^2 deterministically.
// Tangent: the element matrices into a workspace, then a warp per block row
// adds its node's elements in colour order into the block-CSR values.
#include <algorithm>
#include <cmath>

#include "fe_element.cuh"

// ---------------------------------------------------------------- residual
static FollowerFaces follower_faces(fe_mesh m) {
  return FollowerFaces{m->nff, m->ff_nodes, m->ff_kind, m->ff_data, m->fn_ptr, m->fn_list, m->fk_ptr, m->fk_list,
                       m->X};
}

// One thread per element (P1, and P2 meshes of more than RES_ELEMS_PER_SM
// elements per SM): every quadrature point of the element in turn, FP64.  The FP64
// pipe bounds it (one warp instruction holds its SM quarter 64 cycles), so the
// work is counted in FP64 instructions: F comes from differences of the
// derivatives d u / d lambda_k along the barycentric coordinates and the
// nodal forces from P G_k, k = 0..3.  P2: with lambda_k(q) = beta + (alpha -
// beta) delta_kq both split into a part common to the four points and one
// product per k, about 900 FP64 instructions per element where four lanes
// that repeat the shape gradients of ten nodes and add 30 forces across
// lanes take 2,100.  The fibre law works on F in the fibre frame (strains,
// stress and the active tension are products of its columns): 350
// instructions per P1 element instead of 650.  Cook P2 64x64x8 (196k elements)
// 327 us, before 650; 149,760 P1 tets of the fibre law 104 us, before 170.
//
// qp_forces: PG[k][i] = w sum_J P_iJ G_kJ, k = 1..3, and J at one point.  At
// rest (F = I) the terms of the isochoric laws cancel exactly.
template <int KIND>
__device__ __forceinline__ void qp_forces(const MatParams& mp, const double* __restrict__ fib, const double (&F)[9],
                                          double p, const double (&G)[3][3], double w, double (&PG)[3][3], double& J) {
  double c[9];  // cofactor matrix
  c[0] = F[4] * F[8] - F[5] * F[7];
  c[1] = F[5] * F[6] - F[3] * F[8];
  c[2] = F[3] * F[7] - F[4] * F[6];
  c[3] = F[2] * F[7] - F[1] * F[8];
  c[4] = F[0] * F[8] - F[2] * F[6];
  c[5] = F[1] * F[6] - F[0] * F[7];
  c[6] = F[1] * F[5] - F[2] * F[4];
  c[7] = F[2] * F[3] - F[0] * F[5];
  c[8] = F[0] * F[4] - F[1] * F[3];
  J = F[0] * c[0] + F[1] * c[1] + F[2] * c[2];
  if (KIND == FE_MAT_GUCCIONE) {
    double Fr[3][3], fr[9];  // F f_alpha (columns of F in the fibre frame)
#pragma unroll
    for (int q = 0; q < 9; q++) fr[q] = fib[q];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int al = 0; al < 3; al++)
        Fr[i][al] = F[3 * i] * fr[3 * al] + F[3 * i + 1] * fr[3 * al + 1] + F[3 * i + 2] * fr[3 * al + 2];
    // E_ab = (F f_a . F f_b - f_a . f_b) / 2, S'_ab = C e^Q B_ab E_ab
    double S[3][3], Q = 0.0;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = a; b < 3; b++) {
        const double B = a == 0 ? (b == 0 ? mp.bf : mp.bfs) : mp.bt;
        const double E = 0.5 * ((Fr[0][a] * Fr[0][b] + Fr[1][a] * Fr[1][b] + Fr[2][a] * Fr[2][b]) -
                                (fr[3 * a] * fr[3 * b] + fr[3 * a + 1] * fr[3 * b + 1] + fr[3 * a + 2] * fr[3 * b + 2]));
        const double BE = B * E;
        Q += (a == b ? 1.0 : 2.0) * BE * E;
        S[a][b] = S[b][a] = BE;
      }
    const double ce = w * mp.C * exp(Q);
    const double phiJ = w * 0.5 * mp.kappa * (J * log(J) + (J - 1.0)) / J;  // phi / J, phi = kappa/2 (J ln J + J - 1)
    const double an = sqrt(Fr[0][0] * Fr[0][0] + Fr[1][0] * Fr[1][0] + Fr[2][0] * Fr[2][0]);
    const double act = w * mp.gamma / an;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      double gr[3], sg[3];
#pragma unroll
      for (int al = 0; al < 3; al++) gr[al] = fr[3 * al] * G[k][0] + fr[3 * al + 1] * G[k][1] + fr[3 * al + 2] * G[k][2];
#pragma unroll
      for (int a = 0; a < 3; a++) sg[a] = ce * (S[a][0] * gr[0] + S[a][1] * gr[1] + S[a][2] * gr[2]);
      sg[0] += act * gr[0];
#pragma unroll
      for (int i = 0; i < 3; i++)
        PG[k][i] = Fr[i][0] * sg[0] + Fr[i][1] * sg[1] + Fr[i][2] * sg[2] +
                   phiJ * (c[3 * i] * G[k][0] + c[3 * i + 1] * G[k][1] + c[3 * i + 2] * G[k][2]);
    }
    return;
  }
  const double iJ = 1.0 / J;
  double P[9];
  if (KIND == FE_MAT_COOK_NH) {
    double I1 = 0.0;
#pragma unroll
    for (int q = 0; q < 9; q++) I1 += F[q] * F[q];
    const double r = rcbrt(J);
    const double c1 = w * mp.mu * (r * r);
    const double c2 = (w * 2.0 * mp.cvol * (J * J - 1.0) - c1 * (I1 * (1.0 / 3.0))) * iJ;
#pragma unroll
    for (int q = 0; q < 9; q++) P[q] = c1 * F[q] + c2 * c[q];
  } else if (KIND == FE_MAT_TH_NH) {
    const double c1 = w * mp.mu, c2 = -w * (mp.mu + p * J) * iJ;
#pragma unroll
    for (int q = 0; q < 9; q++) P[q] = c1 * F[q] + c2 * c[q];
  } else {  // P = 2a F + 2b F (tr C I - C) - (c + p J) H
    double Cm[9];
    poly_C(F, Cm);
    const double I1 = Cm[0] + Cm[4] + Cm[8], ch = (mp.clog + p * J) * iJ;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const double fc = F[3 * i] * Cm[j] + F[3 * i + 1] * Cm[3 + j] + F[3 * i + 2] * Cm[6 + j];
        P[3 * i + j] = w * (2.0 * mp.ap * F[3 * i + j] + 2.0 * mp.bp * (I1 * F[3 * i + j] - fc) - ch * c[3 * i + j]);
      }
  }
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int i = 0; i < 3; i++) PG[k][i] = P[3 * i] * G[k][0] + P[3 * i + 1] * G[k][1] + P[3 * i + 2] * G[k][2];
}

template <int ORDER, bool MASS, int KIND>
__global__ void __launch_bounds__(128) k_elem_forces(int ne, const int* __restrict__ conn,
                                                     const double* __restrict__ geo, const double* __restrict__ d,
                                                     int nn, int pres, MatParams mp, const double* __restrict__ fib,
                                                     double mass_c, double* __restrict__ rel,
                                                     double* __restrict__ relp) {
  constexpr int NEN = ORDER == 1 ? 4 : 10;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const int* c = conn + (size_t)e * NEN;
  double u[NEN][3], G[3][3];
#pragma unroll
  for (int a = 0; a < NEN; a++) {
    const double* ua = d + 3 * (size_t)c[a];
#pragma unroll
    for (int i = 0; i < 3; i++) u[a][i] = ua[i];
  }
  const double* g = geo + (size_t)e * 10;
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int i = 0; i < 3; i++) G[k][i] = g[3 * k + i];
  const double vol = g[9];
  const double* fe = KIND == FE_MAT_GUCCIONE ? fib + (size_t)e * 9 : nullptr;
  double* out = rel + (size_t)e * NEN * 3;
  if constexpr (ORDER == 1) {
    double F[9], PG[3][3], J;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      double du[3];
#pragma unroll
      for (int k = 0; k < 3; k++) du[k] = u[k + 1][i] - u[0][i];
#pragma unroll
      for (int j = 0; j < 3; j++)
        F[3 * i + j] = (i == j ? 1.0 : 0.0) + du[0] * G[0][j] + du[1] * G[1][j] + du[2] * G[2][j];
    }
    qp_forces<KIND>(mp, fe, F, 0.0, G, vol, PG, J);
#pragma unroll
    for (int i = 0; i < 3; i++) {
      double r[4] = {-(PG[0][i] + PG[1][i] + PG[2][i]), PG[0][i], PG[1][i], PG[2][i]};
      if (MASS) {
        const double mc = mass_c * vol * 0.05, su = (u[0][i] + u[1][i]) + (u[2][i] + u[3][i]);
#pragma unroll
        for (int a = 0; a < 4; a++) r[a] += mc * (su + u[a][i]);
      }
#pragma unroll
      for (int a = 0; a < 4; a++) out[3 * a + i] = r[a];
    }
    return;
  } else {
    constexpr double al = 0.5854101966249685, be = 0.1381966011250105;
    constexpr double uv = 4.0 * be - 1.0, ue = 4.0 * be, dl = 4.0 * (al - be);
    // node of the edge between vertices k and l
    constexpr int ed[4][4] = {{0, 4, 5, 6}, {4, 0, 7, 8}, {5, 7, 0, 9}, {6, 8, 9, 0}};
    double b[4][3];  // d u / d lambda_k without its delta_kq part
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int i = 0; i < 3; i++) {
        double s = 0.0;
#pragma unroll
        for (int l = 0; l < 4; l++)
          if (l != k) s += u[ed[k][l]][i];
        b[k][i] = uv * u[k][i] + ue * s;
      }
    double pv[4] = {0.0, 0.0, 0.0, 0.0}, ps = 0.0;
    if (pres == 1) {
#pragma unroll
      for (int v = 0; v < 4; v++) {
        pv[v] = d[3 * (size_t)nn + c[v]];
        ps += pv[v];
      }
    } else if (pres == 2) {
      ps = d[3 * (size_t)nn + e];
    }
    const double w = 0.25 * vol;
    double r[NEN][3], T[4][3], Jm[4];
#pragma unroll
    for (int a = 0; a < NEN; a++) r[a][0] = r[a][1] = r[a][2] = 0.0;
#pragma unroll
    for (int k = 0; k < 4; k++) T[k][0] = T[k][1] = T[k][2] = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      double F[9], PG[3][3];
#pragma unroll
      for (int i = 0; i < 3; i++) {
        double D[4];
#pragma unroll
        for (int k = 0; k < 4; k++) D[k] = b[k][i] + dl * u[k == q ? q : ed[k][q]][i];
#pragma unroll
        for (int k = 1; k < 4; k++) D[k] -= D[0];
#pragma unroll
        for (int j = 0; j < 3; j++)
          F[3 * i + j] = (i == j ? 1.0 : 0.0) + D[1] * G[0][j] + D[2] * G[1][j] + D[3] * G[2][j];
      }
      const double p = pres == 1 ? be * ps + (al - be) * pv[q] : ps;
      double J;
      qp_forces<KIND>(mp, fe, F, p, G, w, PG, J);
      Jm[q] = J - 1.0;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        const double f[4] = {-(PG[0][i] + PG[1][i] + PG[2][i]), PG[0][i], PG[1][i], PG[2][i]};
#pragma unroll
        for (int k = 0; k < 4; k++) {
          T[k][i] += f[k];
          r[k == q ? q : ed[k][q]][i] += dl * f[k];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
#pragma unroll
      for (int k = 0; k < 4; k++) {
        r[k][i] += uv * T[k][i];
#pragma unroll
        for (int l = k + 1; l < 4; l++) r[ed[k][l]][i] += ue * (T[k][i] + T[l][i]);
      }
      if (MASS) {  // consistent mass through vertex, edge and per-vertex edge sums (mass_hat times 420)
        const double mc = mass_c * vol * (1.0 / 420.0);
        const double sv = (u[0][i] + u[1][i]) + (u[2][i] + u[3][i]);
        double E[4], se = 0.0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
          E[k] = 0.0;
#pragma unroll
          for (int l = 0; l < 4; l++)
            if (l != k) E[k] += u[ed[k][l]][i];
          se += 0.5 * E[k];
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
          r[k][i] += mc * (sv + 5.0 * u[k][i] - 6.0 * se + 2.0 * E[k]);
#pragma unroll
          for (int l = k + 1; l < 4; l++)
            r[ed[k][l]][i] += mc * (2.0 * (u[k][i] + u[l][i]) - 6.0 * sv + 8.0 * (se + E[k] + E[l] + u[ed[k][l]][i]));
        }
      }
#pragma unroll
      for (int a = 0; a < NEN; a++) out[3 * a + i] = r[a][i];
    }
    if (pres) {  // R_p = -int (J - 1) q_h: P1 slots per vertex, P0 all in slot 0
      const double js = (Jm[0] + Jm[1]) + (Jm[2] + Jm[3]);
#pragma unroll
      for (int v = 0; v < 4; v++)
        relp[(size_t)e * 4 + v] = pres == 1 ? -w * (be * js + (al - be) * Jm[v]) : (v == 0 ? -w * js : 0.0);
    }
  }
}

// P2 meshes of fewer elements: a thread per (element, quadrature point).  The
// element thread's chain of four points is the longer one there (whole residual,
// Cook and twist P2: 3,072 elements 40 against 51 us, 6,000 to 6,144: 55-56
// against 51-54, 12,000: 72 against 55, 49,152: 203 against 118; P1 768: 35
// against 29, 96,000: 62 against 53).
constexpr int RES_ELEMS_PER_SM = 40;
template <int ORDER, bool MASS>
__global__ void __launch_bounds__(128) k_elem_residual(int ne, const int* __restrict__ conn,
                                                       const double* __restrict__ geo,
                                                       const double* __restrict__ d, int nn, int pres,
                                                       MatParams mp, const double* __restrict__ fib,
                                                       double mass_c, double* __restrict__ rel,
                                                       double* __restrict__ relp) {
  elem_residual_item<ORDER, MASS>(blockIdx.x * blockDim.x + threadIdx.x, ne, conn, geo, d, nn, pres, mp, fib, mass_c, rel, relp);
}

// Node-wise gather of the element contributions plus the boundary and
// Newmark terms: R = sum rel - load fext1 + Ks d + follower forces - fdyn
// (fdyn = 4/dt^2 M dhat + 2/dt C dtil, nullptr when static; the dashpots'
// 2/dt C d sits in ks_val while dynamics is on).  FOLLOW: the mesh has
// follower faces (the instantiation without them keeps the plain gather's
// registers).
template <int ORDER, bool FOLLOW>
__global__ void __launch_bounds__(256) k_gather_residual(
    int nn, int nen, const int* __restrict__ node_ptr, const int* __restrict__ node_list,
    const double* __restrict__ rel, const double* __restrict__ fext1, double load,
    const int* __restrict__ ks_ptr, const int* __restrict__ ks_col, const double* __restrict__ ks_val,
    const double* __restrict__ d, const uint8_t* __restrict__ fixmask, int np,
    const int* __restrict__ vert_ptr, const int* __restrict__ vert_list, const double* __restrict__ relp,
    FollowerFaces ff, const double* __restrict__ fdyn,
    double* __restrict__ r, double* red, unsigned* ticket, double* norm2, int64_t nrel) {
  const double acc = gather_node<ORDER, FOLLOW>(blockIdx.x * blockDim.x + threadIdx.x, nn, nen, node_ptr, node_list, rel, fext1, load, ks_ptr, ks_col, ks_val, d, fixmask, np, vert_ptr, vert_list, relp, ff, fdyn, r, nrel);
  if (norm2) grid_sum_finish(acc, red, ticket, norm2);
}

template <int ORDER, bool MASS>
static int launch_forces(fe_mesh m, const double* d) {
  auto kern = m->mp.kind == FE_MAT_COOK_NH      ? k_elem_forces<ORDER, MASS, FE_MAT_COOK_NH>
              : m->mp.kind == FE_MAT_TH_NH      ? k_elem_forces<ORDER, MASS, FE_MAT_TH_NH>
              : m->mp.kind == FE_MAT_POLYCONVEX ? k_elem_forces<ORDER, MASS, FE_MAT_POLYCONVEX>
                                                : k_elem_forces<ORDER, MASS, FE_MAT_GUCCIONE>;
  kern<<<(m->ne + 127) / 128, 128, 0, m->stream>>>(m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib,
                                                   m->mass_c, m->rel, m->relp);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

int fe_residual_dev(fe_mesh m, const double* d, double* r, bool want_norm) {
  int nthr = m->ne * m->nq;
  double eb = (double)m->ne * (4.0 * m->nen + 80.0 + 24.0 * m->nen + (m->fib ? 72.0 : 0.0) + (m->pres ? 32.0 : 0.0)) +
              8.0 * (double)m->ndof;
  {
    FE_SCOPE(m, FE_PROF_RESIDUAL, eb);
    const bool dyn = m->dyn != nullptr;
    if (m->order == 1) {
      FE_TRY((dyn ? launch_forces<1, true>(m, d) : launch_forces<1, false>(m, d)));
    } else if (m->ne >= (int64_t)RES_ELEMS_PER_SM * m->sm_count) {
      FE_TRY((dyn ? launch_forces<2, true>(m, d) : launch_forces<2, false>(m, d)));
    } else {
      auto kern = dyn ? k_elem_residual<2, true> : k_elem_residual<2, false>;
      kern<<<(nthr + 127) / 128, 128, 0, m->stream>>>(m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib,
                                                      m->mass_c, m->rel, m->relp);
    }
  }
  FE_CUDA(cudaGetLastError());
  int rows = m->nn + m->np;
  int grid = (rows + 255) / 256;
  if (grid > RED_SLOTS) return fe_set_error("mesh too large for the reduction buffer"), FE_ERR_ARG;
  double gb = (double)m->ne * m->nen * 28.0 + 4.0 * (m->nn + 1) + 25.0 * m->nn + 8.0 * (double)m->ndof +
              (m->pres ? (double)m->ne * 4 * 12.0 + 4.0 * (m->np + 1) : 0.0);
  if (m->dyn) gb += 24.0 * m->nn;
  FE_SCOPE(m, FE_PROF_RESIDUAL, gb);
  const double* fdyn = m->dyn ? m->dyn + 5 * 3 * (size_t)m->nn : nullptr;
  const bool fol = m->nff > 0;
  auto gather = m->order == 1 ? (fol ? k_gather_residual<1, true> : k_gather_residual<1, false>)
                              : (fol ? k_gather_residual<2, true> : k_gather_residual<2, false>);
  gather<<<grid, 256, 0, m->stream>>>(m->nn, m->nen, m->node_ptr, m->node_list, m->rel, m->fext1, m->load,
                                      m->ks_ptr, m->ks_col, m->ks_val, d, m->fixmask, m->np, m->vert_ptr,
                                      m->vert_list, m->relp, follower_faces(m), fdyn, r, m->red, m->red_ticket,
                                      want_norm ? m->scal : nullptr, (int64_t)m->ne * m->nen);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// ---------------------------------------------------------------- energy
template <int ORDER>
__global__ void __launch_bounds__(128) k_elem_energy(int ne, const int* __restrict__ conn,
                                                     const double* __restrict__ geo, const double* __restrict__ d,
                                                     int nn, int pres, MatParams mp, const double* __restrict__ fib,
                                                     double mass_c, double* red, unsigned* ticket, double* out) {
  constexpr int NEN = ORDER == 1 ? 4 : 10;
  constexpr int NQ = ORDER == 1 ? 1 : 4;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int e = t / NQ, q = t % NQ;
  double val = 0.0;
  if (e < ne) {
    const int* c = conn + (size_t)e * NEN;
    double G[4][3], vol;
    load_G(geo, e, G, vol);
    double lam[4];
    for (int k = 0; k < 4; k++) lam[k] = lam_q<ORDER>(q, k);
    QPState<double> s;
    for (int k = 0; k < 9; k++) s.F[k] = (k % 4 == 0) ? 1.0 : 0.0;
    for (int a = 0; a < NEN; a++) {
      double g[3];
      shape_grad<ORDER>(a, lam, G, g);
      for (int i = 0; i < 3; i++)
        for (int J = 0; J < 3; J++) s.F[3 * i + J] += d[3 * (size_t)c[a] + i] * g[J];
    }
    s.p = 0.0;
    if (pres == 1)
      for (int v = 0; v < 4; v++) s.p += d[3 * (size_t)nn + c[v]] * lam[v];
    else if (pres == 2)
      s.p = d[3 * (size_t)nn + e];
    const double* fe = fib ? fib + (size_t)e * 9 : nullptr;
    qp_prepare(mp, fe, s);
    val = vol / NQ * qp_energy(mp, s);
    if (mass_c != 0.0 && q == 0)  // inertia of the step: mass_c / 2 d^T M d
      for (int a = 0; a < NEN; a++)
        for (int b = 0; b < NEN; b++) {
          const double* ua = d + 3 * (size_t)c[a];
          const double* ub = d + 3 * (size_t)c[b];
          val += 0.5 * mass_c * vol * mass_hat(ORDER, a, b) * (ua[0] * ub[0] + ua[1] * ub[1] + ua[2] * ub[2]);
        }
  }
  grid_sum_finish(val, red, ticket, out);
}

// boundary part of the energy: -load fext.d + d.Ks d / 2, and -fdyn.d of a
// Newmark step (fdyn nullptr when static)
__global__ void k_node_energy(int nn, const double* __restrict__ fext1, double load, const int* __restrict__ ks_ptr,
                              const int* __restrict__ ks_col, const double* __restrict__ ks_val,
                              const double* __restrict__ fdyn, const double* __restrict__ d, double* red,
                              unsigned* ticket, double* out) {
  int a = blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (a < nn) {
    const double* u = d + 3 * (size_t)a;
    v = -load * (fext1[3 * a] * u[0] + fext1[3 * a + 1] * u[1] + fext1[3 * a + 2] * u[2]);
    if (fdyn) v -= fdyn[3 * (size_t)a] * u[0] + fdyn[3 * (size_t)a + 1] * u[1] + fdyn[3 * (size_t)a + 2] * u[2];
    for (int k = ks_ptr[a]; k < ks_ptr[a + 1]; k++) {
      const double* kv = ks_val + (size_t)k * 9;
      const double* w = d + 3 * (size_t)ks_col[k];
      for (int i = 0; i < 3; i++) v += 0.5 * u[i] * (kv[3 * i] * w[0] + kv[3 * i + 1] * w[1] + kv[3 * i + 2] * w[2]);
    }
  }
  grid_sum_finish(v, red, ticket, out);
}

int fe_energy_dev(fe_mesh m, const double* d, double* out) {
  int nthr = m->ne * m->nq;
  int grid = (nthr + 127) / 128;
  if (grid > RED_SLOTS) {
    // large meshes: the element sum in two halves would change the order; keep one pass
    return fe_set_error("mesh too large for the energy reduction"), FE_ERR_ARG;
  }
  const double mass_c = m->dyn ? m->mass_c : 0.0;
  if (m->order == 1)
    k_elem_energy<1><<<grid, 128, 0, m->stream>>>(m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib,
                                                  mass_c, m->red, m->red_ticket, m->scal + 1);
  else
    k_elem_energy<2><<<grid, 128, 0, m->stream>>>(m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib,
                                                  mass_c, m->red, m->red_ticket, m->scal + 1);
  FE_CUDA(cudaGetLastError());
  const double* fdyn = m->dyn ? m->dyn + 5 * 3 * (size_t)m->nn : nullptr;
  k_node_energy<<<(m->nn + 255) / 256, 256, 0, m->stream>>>(m->nn, m->fext1, m->load, m->ks_ptr, m->ks_col,
                                                            m->ks_val, fdyn, d, m->red, m->red_ticket, m->scal + 2);
  FE_CUDA(cudaGetLastError());
  FE_CUDA(cudaMemcpyAsync(m->h_scal + 1, m->scal + 1, 2 * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  *out = m->h_scal[1] + m->h_scal[2] + (m->dyn ? m->dyn_const : 0.0);
  return FE_OK;
}

// ---------------------------------------------------------------- tangent
// Two kernels.  k_elem_blocks64 / k_elem_blocks32 compute every element's
// matrix once (blocks (a, b), a <= b; the tangent of a potential is symmetric)
// into a workspace; k_gather_tangent adds, one warp per block row, the
// contributions of the node's elements in colour order and writes the finished
// row in the tiled layout.  Each block is written once, in 128-byte runs.
// (Before: one launch per colour, elements spread over a block's threads,
// scattered 4-byte read-modify-writes, each its own 32-byte sector of eight.
// Cook P2 45x41x7 in FP32: 38 launches, 1,580 us; now 171 + 183 us, the blocks
// 23 us of traffic at the copy rate each way.  Cardiac shell of 149,760 P1 tets
// in FP64: 3.1 ms; now 486 us, bound by the FP64 pipe, + 148 us.)  A mesh whose
// workspace does not fit is assembled colour by colour (k_elem_tangent).
//
// FP64: at a quadrature point the material tangent A enters the element matrix
// only through the four barycentric gradients G_k: M_kl[i][j] = sum_JL G_kJ
// A_iJjL G_lL, k, l = 0..3.  qp_blocks forms M from the law's own terms (F G_k,
// H G_k, fibre-frame strains of the directions e_i x G_k), 6 pairs of 9 values,
// without the 81 entries of A (for the fibre law about a sixth of the FP64
// operations, which bound it); the pairs with G_0 = -(G_1 + G_2 + G_3) follow
// by sums.  P1: K_ab = w M_ab.  P2: K_ab = sum_q w sum_kl c_ak(q) c_bl(q)
// M_kl(q) with at most two k per node and coefficients that depend on q only
// through lambda_k(q) = beta + (alpha - beta) delta_kq.
__device__ __forceinline__ constexpr int pair4(int k, int l) {  // k <= l < 4
  return k * 4 - k * (k - 1) / 2 + (l - k);
}

template <class T>
__device__ void qp_blocks(const MatParams& mp, const double* __restrict__ fib, const QPState<T>& s, const T (*G)[3],
                          T* __restrict__ M) {
  const T* F = s.F;
  const T* H = s.H;
  T FG[3][3], HG[3][3];  // [k - 1][i]
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int i = 0; i < 3; i++) {
      FG[k][i] = F[3 * i] * G[k + 1][0] + F[3 * i + 1] * G[k + 1][1] + F[3 * i + 2] * G[k + 1][2];
      HG[k][i] = H[3 * i] * G[k + 1][0] + H[3 * i + 1] * G[k + 1][1] + H[3 * i + 2] * G[k + 1][2];
    }
  auto put = [&](int k, int l, int i, int j, T v) { M[9 * pair4(k + 1, l + 1) + 3 * i + j] = v; };
  if (mp.kind == FE_MAT_COOK_NH) {
    const T j13 = dcbrt(s.J);
    const T mj = (T)mp.mu / (j13 * j13), cv = (T)mp.cvol, J2 = s.J * s.J;
    const T c23 = -mj * (T(2) / T(3)), chh = mj * (T(2) / T(9)) * s.I1 + T(4) * cv * J2,
            cht = mj * s.I1 / T(3) - T(2) * cv * (J2 - T(1));
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
      for (int l = k; l < 3; l++) {
        const T gg = mj * (G[k + 1][0] * G[l + 1][0] + G[k + 1][1] * G[l + 1][1] + G[k + 1][2] * G[l + 1][2]);
#pragma unroll
        for (int i = 0; i < 3; i++) {
          const T ah = c23 * FG[k][i] + chh * HG[k][i], af = c23 * HG[k][i], at = cht * HG[l][i];
#pragma unroll
          for (int j = 0; j < 3; j++)
            put(k, l, i, j, ah * HG[l][j] + af * FG[l][j] + at * HG[k][j] + (i == j ? gg : T(0)));
        }
      }
  } else if (mp.kind == FE_MAT_TH_NH) {
    const T mu = (T)mp.mu, pJ = s.p * s.J;
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
      for (int l = k; l < 3; l++) {
        const T gg = mu * (G[k + 1][0] * G[l + 1][0] + G[k + 1][1] * G[l + 1][1] + G[k + 1][2] * G[l + 1][2]);
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
          for (int j = 0; j < 3; j++)
            put(k, l, i, j, (mu + pJ) * (HG[l][i] * HG[k][j]) - pJ * (HG[k][i] * HG[l][j]) + (i == j ? gg : T(0)));
      }
  } else if (mp.kind == FE_MAT_POLYCONVEX) {
    const T a = (T)mp.ap, b = (T)mp.bp, c = (T)mp.clog, pJ = s.p * s.J;
    T Bm[9];  // F F^T
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = 0; j < 3; j++)
        Bm[3 * i + j] = F[3 * i] * F[3 * j] + F[3 * i + 1] * F[3 * j + 1] + F[3 * i + 2] * F[3 * j + 2];
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
      for (int l = k; l < 3; l++) {
        const T gg = G[k + 1][0] * G[l + 1][0] + G[k + 1][1] * G[l + 1][1] + G[k + 1][2] * G[l + 1][2];
        const T ff = FG[k][0] * FG[l][0] + FG[k][1] * FG[l][1] + FG[k][2] * FG[l][2];
        const T dg = T(2) * a * gg + T(2) * b * (s.I1 * gg - ff);
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
          for (int j = 0; j < 3; j++)
            put(k, l, i, j,
                T(2) * b * (T(2) * FG[l][j] * FG[k][i] - FG[l][i] * FG[k][j] - Bm[3 * i + j] * gg) +
                    (c + pJ) * (HG[l][i] * HG[k][j]) - pJ * (HG[k][i] * HG[l][j]) + (i == j ? dg : T(0)));
      }
  } else {
    T fr[9];  // rows f, s, n
#pragma unroll
    for (int q = 0; q < 9; q++) fr[q] = (T)fib[q];
    T Fr[9], Gr[3][3];  // rows of F and the gradients in the fibre frame
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int al = 0; al < 3; al++) {
        Fr[3 * i + al] = F[3 * i] * fr[3 * al] + F[3 * i + 1] * fr[3 * al + 1] + F[3 * i + 2] * fr[3 * al + 2];
        Gr[i][al] = fr[3 * al] * G[i + 1][0] + fr[3 * al + 1] * G[i + 1][1] + fr[3 * al + 2] * G[i + 1][2];
      }
    const T ce = (T)mp.C * s.eQ;
    // strain of the direction e_i x G_k: (ff, ss, nn, fs, fn, sn), and D : dE
    T E[3][3][6], d[3][3], SG[3][3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      T DG[3];
#pragma unroll
      for (int q = 0; q < 3; q++) {
        DG[q] = s.D[3 * q] * G[k + 1][0] + s.D[3 * q + 1] * G[k + 1][1] + s.D[3 * q + 2] * G[k + 1][2];
        SG[k][q] = ce * DG[q];  // S = C e^Q D
      }
#pragma unroll
      for (int i = 0; i < 3; i++) {
        const T* f = Fr + 3 * i;
        const T* g = Gr[k];
        E[k][i][0] = f[0] * g[0];
        E[k][i][1] = f[1] * g[1];
        E[k][i][2] = f[2] * g[2];
        E[k][i][3] = T(0.5) * (f[0] * g[1] + g[0] * f[1]);
        E[k][i][4] = T(0.5) * (f[0] * g[2] + g[0] * f[2]);
        E[k][i][5] = T(0.5) * (f[1] * g[2] + g[1] * f[2]);
        d[k][i] = F[3 * i] * DG[0] + F[3 * i + 1] * DG[1] + F[3 * i + 2] * DG[2];
      }
    }
    const T bf = (T)mp.bf, bt = (T)mp.bt, bfs = (T)mp.bfs;
    const T wt[6] = {ce * bf, ce * bt, ce * bt, T(2) * ce * bfs, T(2) * ce * bfs, T(2) * ce * bt};
    const T lJ = dlog(s.J);
    const T phi = T(0.5) * (T)mp.kappa * (s.J * lJ + s.J - T(1));
    const T dphiJ = T(0.5) * (T)mp.kappa * (lJ + T(2)) * s.J;
    const T ga = (T)mp.gamma / s.an, ian2 = T(1) / (s.an * s.an);
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
      for (int l = k; l < 3; l++) {
        const T act = ga * Gr[k][0] * Gr[l][0];
        const T gsg = G[l + 1][0] * SG[k][0] + G[l + 1][1] * SG[k][1] + G[l + 1][2] * SG[k][2];
#pragma unroll
        for (int i = 0; i < 3; i++) {
          T we[6];
#pragma unroll
          for (int q = 0; q < 6; q++) we[q] = wt[q] * E[k][i][q];
          const T dd = T(2) * ce * d[k][i], dh = dphiJ * HG[k][i], ph = phi * HG[l][i], aa = act * s.a[i] * ian2;
#pragma unroll
          for (int j = 0; j < 3; j++) {
            T v = dd * d[l][j] + dh * HG[l][j] - ph * HG[k][j] - aa * s.a[j];
#pragma unroll
            for (int q = 0; q < 6; q++) v += we[q] * E[l][j][q];
            put(k, l, i, j, v + (i == j ? gsg + act : T(0)));
          }
        }
      }
  }
  // pairs with G_0: M_0l = -(M_1l + M_2l + M_3l), M_00 = -(M_10 + M_20 + M_30)
  auto get = [&](int k, int l, int i, int j) { return k <= l ? M[9 * pair4(k, l) + 3 * i + j] : M[9 * pair4(l, k) + 3 * j + i]; };
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
      for (int l = 1; l < 4; l++)
        M[9 * pair4(0, l) + 3 * i + j] = -(get(1, l, i, j) + get(2, l, i, j) + get(3, l, i, j));
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++)
      M[3 * i + j] = -(M[9 * pair4(0, 1) + 3 * j + i] + M[9 * pair4(0, 2) + 3 * j + i] + M[9 * pair4(0, 3) + 3 * j + i]);
}

template <int ORDER>
struct Blk64Cfg {
  static constexpr int NEN = ORDER == 1 ? 4 : 10;
  static constexpr int NQ = ORDER == 1 ? 1 : 4;
  static constexpr int NPAIR = NEN * (NEN + 1) / 2;
  static constexpr int EB = ORDER == 1 ? 64 : 16;      // elements per block
  static constexpr int THREADS = ORDER == 1 ? 64 : 144;  // P2: one per (element, block entry) in the second phase
  static constexpr int MS = 91;                         // stride of a point's M (odd: no bank conflicts)
};

// FP64: the element's blocks (a, b), a <= b, [NPAIR][9], and the u-p coupling
// [NEN][npl][3]; inertia (mass_c M) included
template <int ORDER, class T>
__global__ void __launch_bounds__(Blk64Cfg<ORDER>::THREADS)
    k_elem_blocks64(int ne, const int* __restrict__ conn, const double* __restrict__ geo, const double* __restrict__ d,
                  int nn, int pres, MatParams mp, const double* __restrict__ fib, double mass_c, T* __restrict__ Ke,
                  T* __restrict__ Be) {
  using C = Blk64Cfg<ORDER>;
  constexpr int NEN = C::NEN, NQ = C::NQ, EB = C::EB, MS = C::MS;
  extern __shared__ __align__(16) unsigned char smraw[];
  T* Ms = reinterpret_cast<T*>(smraw);   // [EB * NQ][MS]
  T* Hs = Ms + EB * NQ * MS;             // u-p: [EB * NQ][12] -J H G_k
  __shared__ T vols[EB];
  const int e0 = blockIdx.x * EB;
  const int eb = min(EB, ne - e0);
  for (int t = threadIdx.x; t < eb * NQ; t += blockDim.x) {
    const int e = e0 + t / NQ, q = t % NQ;
    T G[4][3], vol, lam[4];
    QPState<T> s;
    qp_point<ORDER, T>(e, q, conn + (size_t)e * NEN, geo, d, nn, pres, mp, fib, s, G, lam, vol, [](int, const T (&)[3]) {});
    qp_blocks<T>(mp, fib ? fib + (size_t)e * 9 : nullptr, s, G, Ms + t * MS);
    if (pres)
#pragma unroll
      for (int k = 0; k < 4; k++)
#pragma unroll
        for (int i = 0; i < 3; i++)
          Hs[t * 12 + 3 * k + i] = -s.J * (s.H[3 * i] * G[k][0] + s.H[3 * i + 1] * G[k][1] + s.H[3 * i + 2] * G[k][2]);
    if (q == 0) vols[t / NQ] = vol;
  }
  __syncthreads();
  if (ORDER == 1) {  // K_ab = vol M_ab, written in the elements' order
    for (int t = threadIdx.x; t < eb * 90; t += blockDim.x) {
      const int le = t / 90, r = t - le * 90, ij = r % 9;
      T v = vols[le] * Ms[le * MS + r];
      if (mass_c != 0.0 && ij % 4 == 0) {
        const int p = r / 9, a = p < 4 ? 0 : (p < 7 ? 1 : (p < 9 ? 2 : 3)), b = p - pair4(a, a) + a;
        v += (T)(mass_c * (double)vols[le] * mass_hat(1, a, b));
      }
      Ke[(size_t)(e0 + le) * 90 + r] = v;
    }
    return;
  }
  // P2: thread (element, entry ij), the 16 ordered barycentric pairs of its
  // entry at the four points in registers
  constexpr int ep[6] = {0, 0, 0, 1, 1, 2}, eq[6] = {1, 2, 3, 2, 3, 3};
  const int le = threadIdx.x / 9, ij = threadIdx.x % 9, ji = 3 * (ij % 3) + ij / 3;
  if (le < eb) {
    const T w = vols[le] / T(NQ);
    T m[4][4][4], S[4][4];  // [q][k][l], sum over q
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int l = 0; l < 4; l++) {
#pragma unroll
        for (int q = 0; q < 4; q++)
          m[q][k][l] = w * Ms[(le * 4 + q) * MS + (k <= l ? 9 * pair4(k, l) + ij : 9 * pair4(l, k) + ji)];
        S[k][l] = (m[0][k][l] + m[1][k][l]) + (m[2][k][l] + m[3][k][l]);
      }
    const double al = 0.5854101966249685, be = 0.1381966011250105;
    const T uv = (T)(4.0 * be - 1.0), ue = (T)(4.0 * be), dl = (T)(4.0 * (al - be));
    // sum_q (u1 + dl [q = s1]) (u2 + dl [q = s2]) m[q][k][l]
    auto term = [&](T u1, int s1, T u2, int s2, int k, int l) -> T {
      if (s1 == s2) return u1 * u2 * S[k][l] + dl * (u1 + u2 + dl) * m[s1][k][l];
      return u1 * u2 * S[k][l] + dl * u1 * m[s2][k][l] + dl * u2 * m[s1][k][l];
    };
    T* out = Ke + (size_t)(e0 + le) * (C::NPAIR * 9) + ij;
    const bool mass = mass_c != 0.0 && ij % 4 == 0;
    const double mv = mass ? mass_c * (double)vols[le] : 0.0;
    int pr = 0;
#pragma unroll
    for (int a = 0; a < 10; a++)
#pragma unroll
      for (int b = a; b < 10; b++) {
        T v;
        if (b < 4) {
          v = term(uv, a, uv, b, a, b);
        } else if (a < 4) {
          const int p = ep[b - 4], r = eq[b - 4];  // node b: 4 (lambda_p G_r + lambda_r G_p)
          v = term(uv, a, ue, p, a, r) + term(uv, a, ue, r, a, p);
        } else {
          const int p = ep[a - 4], r = eq[a - 4], s = ep[b - 4], t = eq[b - 4];
          v = (term(ue, p, ue, s, r, t) + term(ue, p, ue, t, r, s)) + (term(ue, r, ue, s, p, t) + term(ue, r, ue, t, p, s));
        }
        if (mass) v += (T)(mv * mass_hat(2, a, b));
        out[9 * pr] = v;
        pr++;
      }
  }
  // u-p coupling: sum_q w lv(q) sum_J (-J H)_iJ g_aJ over the element's local
  // pressure values (P1: 4 vertices, P0: 1)
  if (pres) {
    const int npl = pres == 2 ? 1 : 4;
    for (int t = threadIdx.x; t < eb * NEN * npl; t += blockDim.x) {
      const int v = t % npl, a = (t / npl) % NEN, l = t / (npl * NEN);
      T acc[3] = {T(0), T(0), T(0)};
      for (int q = 0; q < NQ; q++) {
        const T* h = Hs + (l * NQ + q) * 12;
        const T lv = pres == 2 ? T(1) : (T)lam_q<ORDER>(q, v);
        for (int i = 0; i < 3; i++) {
          T g;
          if (a < 4) g = (T)(4.0 * lam_q<ORDER>(q, a) - 1.0) * h[3 * a + i];
          else
            g = T(4) * ((T)lam_q<ORDER>(q, ep[a - 4]) * h[3 * eq[a - 4] + i] +
                        (T)lam_q<ORDER>(q, eq[a - 4]) * h[3 * ep[a - 4] + i]);
          acc[i] += lv * g;
        }
      }
      const T w = vols[l] / T(NQ);
      for (int i = 0; i < 3; i++) Be[((size_t)(e0 + l) * NEN * npl + a * npl + v) * 3 + i] = w * acc[i];
    }
  }
}

// FP32: the same blocks in the arithmetic of tangent_tile (A per point, C_b =
// A g_b, K_ab = sum_q w g_a C_b), bit for bit: the FP32 V-cycle amplifies the
// rounding of the tangent by the condition of its coarse operators, so the
// values keep their order of operations whichever kernel forms them.  C_b
// stays in registers: a thread takes rows i of the blocks (., b) of its b (P2:
// of b and 9 - b, eleven blocks each), reading A's rows and the gradients from
// shared memory by 16 bytes.
template <int ORDER>
struct Blk32Cfg {
  static constexpr int NEN = ORDER == 1 ? 4 : 10;
  static constexpr int NQ = ORDER == 1 ? 1 : 4;
  static constexpr int NPAIR = NEN * (NEN + 1) / 2;
  static constexpr int EB = 16;                      // elements per block
  static constexpr int TPE = ORDER == 1 ? 12 : 15;   // threads per element
  static constexpr int THREADS = EB * TPE;
  static constexpr int AROW = 28;                    // one i: 27 values of A, padded
  static constexpr int SZ_A = NQ * 3 * AROW, SZ_G = NQ * NEN * 4;
  static constexpr int PER_E = SZ_A + SZ_G + 4;      // floats (the pad spreads the elements over the banks)
};

template <int ORDER>
__global__ void __launch_bounds__(Blk32Cfg<ORDER>::THREADS, 2)
    k_elem_blocks32(int ne, const int* __restrict__ conn, const double* __restrict__ geo, const double* __restrict__ d,
                    int nn, int pres, MatParams mp, const double* __restrict__ fib, double mass_c,
                    float* __restrict__ Ke, float* __restrict__ Be) {
  using C = Blk32Cfg<ORDER>;
  using T = float;
  constexpr int NEN = C::NEN, NQ = C::NQ, EB = C::EB;
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);   // [EB][PER_E]: A [NQ][3][AROW], g [NQ][NEN][4]
  T* dps = sm + EB * C::PER_E;           // u-p: [EB * NQ][9]
  __shared__ QPState<T> qs[EB * NQ];
  __shared__ T ws[EB];
  const int e0 = blockIdx.x * EB, eb = min(EB, ne - e0);
  for (int k = threadIdx.x; k < eb * NQ; k += blockDim.x) {
    const int le = k / NQ, q = k % NQ, e = e0 + le;
    T G[4][3], vol, lam[4];
    T* gb = sm + le * C::PER_E + C::SZ_A + q * NEN * 4;
    QPState<T>& s = qs[k];
    qp_point<ORDER, T>(e, q, conn + (size_t)e * NEN, geo, d, nn, pres, mp, fib, s, G, lam, vol,
                       [&](int a, const T (&g)[3]) {
                         *reinterpret_cast<float4*>(gb + 4 * a) = make_float4(g[0], g[1], g[2], 0.f);
                       });
    if (q == 0) ws[le] = vol / NQ;
    if (pres)
      for (int j = 0; j < 9; j++) dps[k * 9 + j] = -s.J * s.H[j];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < eb * NQ * 9; k += blockDim.x) {
    const int lq = k / 9, kl = k % 9, le = lq / NQ, q = lq % NQ;
    T colv[9];
    qp_tangent_col(mp, fib ? fib + (size_t)(e0 + le) * 9 : nullptr, qs[lq], kl / 3, kl % 3, colv);
    T* A = sm + le * C::PER_E + q * 3 * C::AROW;
#pragma unroll
    for (int ij = 0; ij < 9; ij++) A[(ij / 3) * C::AROW + (ij % 3) * 9 + kl] = colv[ij];
  }
  __syncthreads();
  const int le = threadIdx.x / C::TPE, r = threadIdx.x % C::TPE, i = r % 3;
  if (le < eb) {
    const T* A = sm + le * C::PER_E + i * C::AROW;
    const T* g = sm + le * C::PER_E + C::SZ_A;
    const T w = ws[le];
    T* out = Ke + (size_t)(e0 + le) * (C::NPAIR * 9) + 3 * i;
#pragma unroll 1
    for (int h = 0; h < (ORDER == 1 ? 1 : 2); h++) {
      const int b = h == 0 ? r / 3 : 9 - r / 3;
      T c[NQ][3][3];
#pragma unroll
      for (int q = 0; q < NQ; q++) {
        T a[C::AROW];
#pragma unroll
        for (int t = 0; t < C::AROW / 4; t++)
          *reinterpret_cast<float4*>(a + 4 * t) = *reinterpret_cast<const float4*>(A + q * 3 * C::AROW + 4 * t);
        const float4 gb = *reinterpret_cast<const float4*>(g + (q * NEN + b) * 4);
#pragma unroll
        for (int J = 0; J < 3; J++)
#pragma unroll
          for (int kk = 0; kk < 3; kk++)
            c[q][J][kk] = a[9 * J + 3 * kk] * gb.x + a[9 * J + 3 * kk + 1] * gb.y + a[9 * J + 3 * kk + 2] * gb.z;
      }
#pragma unroll 1
      for (int a = 0; a <= b; a++) {
        T acc[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int q = 0; q < NQ; q++) {
          const float4 g4 = *reinterpret_cast<const float4*>(g + (q * NEN + a) * 4);
          const T ga[3] = {g4.x, g4.y, g4.z};
#pragma unroll
          for (int J = 0; J < 3; J++)
#pragma unroll
            for (int kk = 0; kk < 3; kk++) acc[kk] += ga[J] * c[q][J][kk];
        }
        if (mass_c != 0.0) {  // inertia of a Newmark step: 4 rho / dt^2 M_ab on the block diagonal
          const T mv = (T)(mass_c * NQ * mass_hat(ORDER, a, b));
#pragma unroll
          for (int kk = 0; kk < 3; kk++)
            if (kk == i) acc[kk] += mv;
        }
        T* o = out + 9 * (a * NEN - a * (a - 1) / 2 + (b - a));
#pragma unroll
        for (int kk = 0; kk < 3; kk++) o[kk] = w * acc[kk];
      }
    }
  }
  if (pres) {  // u-p coupling, as in tangent_tile
    const int npl = pres == 2 ? 1 : 4;
    for (int k = threadIdx.x; k < eb * NEN * npl; k += blockDim.x) {
      const int v = k % npl, a = (k / npl) % NEN, l = k / (npl * NEN);
      T acc[3] = {T(0), T(0), T(0)};
      for (int q = 0; q < NQ; q++) {
        const T* dp = dps + (l * NQ + q) * 9;
        const T* ga = sm + l * C::PER_E + C::SZ_A + (q * NEN + a) * 4;
        const T lv = pres == 2 ? T(1) : (T)lam_q<ORDER>(q, v);
        for (int ii = 0; ii < 3; ii++)
          acc[ii] += lv * (dp[3 * ii] * ga[0] + dp[3 * ii + 1] * ga[1] + dp[3 * ii + 2] * ga[2]);
      }
      for (int ii = 0; ii < 3; ii++) Be[(((size_t)(e0 + l) * NEN + a) * npl + v) * 3 + ii] = ws[l] * acc[ii];
    }
  }
}

// One warp per block row: the row's blocks in shared memory (chunks of
// TG_CHUNK blocks), the node's elements in colour order (the next element's
// values are loaded while the current ones are added; a node pair occurs once
// in an element, so its values have distinct places), prescribed rows and
// columns zeroed, then the row into the tiles.
constexpr int TG_CHUNK = 96;
constexpr int TG_WARPS = 4;
template <int ORDER, class T>
__global__ void __launch_bounds__(32 * TG_WARPS)
    k_gather_tangent(int nn, const int* __restrict__ node_ptr, const int* __restrict__ node_list,
                     const int* __restrict__ emap, const T* __restrict__ Ke, const int* __restrict__ row_ptr,
                     const int* __restrict__ col, const uint8_t* __restrict__ fixmask, T* __restrict__ K, int npl,
                     const int* __restrict__ upmap, const T* __restrict__ Be, const int* __restrict__ up_ptr,
                     T* __restrict__ B, int64_t nnzb) {
  using C = Blk64Cfg<ORDER>;  // (the layout of Ke is the same in FP32)
  constexpr int NEN = C::NEN, NV = (NEN * 9 + 31) / 32;
  __shared__ T accs[TG_WARPS][TG_CHUNK * 9];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int row = blockIdx.x * TG_WARPS + wid;
  if (row >= nn) return;
  T* acc = accs[wid];
  const int ls = node_ptr[row], lend = node_ptr[row + 1];
  const int rs = row_ptr[row], re = row_ptr[row + 1];
  const unsigned fr = fixmask[row];
  for (int cb = rs; cb < re; cb += TG_CHUNK) {
    const int m = min(TG_CHUNK, re - cb);
    for (int t = lane; t < m * 9; t += 32) acc[t] = T(0);
    __syncwarp();
    T nv[NV];
    int np[NV];
    auto load = [&](int k) {  // this lane's values of the node's k-th element, and their places
#pragma unroll
      for (int u = 0; u < NV; u++) {
        const int t = lane + 32 * u;
        np[u] = -1;
        if (k < lend && t < NEN * 9) {
          const int slot = node_list[k], e = slot / NEN, a = slot - e * NEN, b = t / 9, ij = t - 9 * b;
          const int lo = min(a, b), hi = max(a, b);
          const int pr = lo * NEN - lo * (lo - 1) / 2 + (hi - lo);
          nv[u] = Ke[(size_t)e * (C::NPAIR * 9) + 9 * pr + (a <= b ? ij : 3 * (ij % 3) + ij / 3)];
          const int pos = fe_idx(emap[(size_t)e * NEN * NEN + a * NEN + b], nnzb) - cb;
          if (pos >= 0 && pos < m) np[u] = 9 * pos + ij;
        }
      }
    };
    load(ls);
    for (int k = ls; k < lend; k++) {
      T cv[NV];
      int cp[NV];
#pragma unroll
      for (int u = 0; u < NV; u++) {
        cv[u] = nv[u];
        cp[u] = np[u];
      }
      load(k + 1);
#pragma unroll
      for (int u = 0; u < NV; u++)
        if (cp[u] >= 0) acc[cp[u]] += cv[u];
      __syncwarp();
    }
    for (int pos = lane; pos < m; pos += 32) {
      const unsigned fc = fixmask[col[cb + pos]];
#pragma unroll
      for (int c = 0; c < 9; c++)
        K[kv_index(cb + pos, c)] = (((fr >> (c / 3)) & 1u) || ((fc >> (c % 3)) & 1u)) ? T(0) : acc[9 * pos + c];
    }
    __syncwarp();
  }
  if (npl) {
    const int us = up_ptr[row], ue = up_ptr[row + 1];
    for (int cb = us; cb < ue; cb += TG_CHUNK) {
      const int m = min(TG_CHUNK, ue - cb);
      for (int t = lane; t < m * 3; t += 32) acc[t] = T(0);
      __syncwarp();
      for (int k = ls; k < lend; k++) {
        const int slot = node_list[k];
        if (lane < npl * 3) {
          const int pos = upmap[(size_t)slot * npl + lane / 3] - cb;
          if (pos >= 0 && pos < m) acc[3 * pos + lane % 3] += Be[((size_t)slot * npl + lane / 3) * 3 + lane % 3];
        }
        __syncwarp();
      }
      for (int t = lane; t < m * 3; t += 32) B[(size_t)cb * 3 + t] = ((fr >> (t % 3)) & 1u) ? T(0) : acc[t];
      __syncwarp();
    }
  }
}

// One CTA assembles EPB elements of one colour into the block-CSR values.
template <int ORDER, class T>
__global__ void __launch_bounds__(256) k_elem_tangent(
    int nel, const int* __restrict__ elems, const int* __restrict__ conn, const double* __restrict__ geo,
    const double* __restrict__ d, int nn, int pres, MatParams mp, const double* __restrict__ fib,
    const int* __restrict__ emap, const int* __restrict__ upmap, const uint8_t* __restrict__ fixmask,
    double mass_c, T* __restrict__ K, T* __restrict__ B, int64_t nnzb) {
  tangent_tile<ORDER, T>(blockIdx.x, nel, elems, conn, geo, d, nn, pres, mp, fib, emap, upmap, fixmask, mass_c, K, B, nnzb);
}

// face-pattern blocks: springs (plus 2/dt dashpots while dynamics is on)
// and the follower-pressure blocks at d, in FP64, prescribed components
// masked; one thread per entry, its faces in a fixed order
template <int ORDER, class T>
__global__ void k_add_face_blocks(int64_t nnz_ks, const int* __restrict__ ks_row, const int* __restrict__ ks_col,
                                  const double* __restrict__ ks_val, const int* __restrict__ ks_kpos,
                                  const uint8_t* __restrict__ fixmask, FollowerFaces ff,
                                  const double* __restrict__ d, double load, T* K) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nnz_ks) face_block_entry<ORDER, T>((int)k, ks_row[k], ks_col, ks_val, ks_kpos, fixmask, ff, d, load, K);
}

// unit diagonal at prescribed components, then invert each 3x3 diagonal block
template <class T, class DT>
__global__ void k_diag_inverse(int nn, const int* __restrict__ diag_pos, const uint8_t* __restrict__ fixmask,
                               T* K, DT* Dinv) {
  diag_inverse_row<T, DT>(blockIdx.x * blockDim.x + threadIdx.x, nn, diag_pos, fixmask, K, Dinv);
}

// SIMPLE Schur diagonal: S_vv = -sum_{(a,v)} sum_i B[a,v]_i^2 / A_(ai,ai), a
// warp per vertex (a thread per vertex walked its 60-odd nodes' three FP64
// divisions alone: 220 us for 2,197 vertices)
template <class T>
__global__ void k_schur_diag(int np, const int* __restrict__ pu_ptr, const int* __restrict__ pu_col,
                             const int* __restrict__ pu_src, const int* __restrict__ diag_pos,
                             const T* __restrict__ K, const T* __restrict__ B, double* Sd) {
  const int v = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (v >= np) return;
  double s = 0.0;
  for (int k = pu_ptr[v] + lane; k < pu_ptr[v + 1]; k += 32) {
    const int p = diag_pos[pu_col[k]];
    const T* b = B + (size_t)pu_src[k] * 3;
    for (int i = 0; i < 3; i++) s -= (double)b[i] * (double)b[i] / (double)K[kv_index(p, 4 * i)];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) Sd[v] = s;
}

__global__ void k_to_bf16(int64_t n, const float* __restrict__ src, __nv_bfloat16* __restrict__ dst) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

// the element blocks' workspace, kept in the mesh (the larger of the two
// precisions it was asked for) until another allocation of the mesh needs the
// memory (fe_alloc); FE_ERR_OOM where it does not fit.  Above
// TAN_WORK_SMALL it takes at most a quarter of the free memory, so that what
// the caller and other meshes allocate next finds the rest (P2 in FP64: 4 kB an
// element, more than the matrix).
constexpr size_t TAN_WORK_SMALL = (size_t)64 << 20;
static int tangent_workspace(fe_mesh m, size_t elem) {
  const size_t npair = (size_t)m->nen * (m->nen + 1) / 2, npl = m->pres == 0 ? 0 : (m->pres == 2 ? 1 : 4);
  const size_t bytes = (size_t)m->ne * (9 * npair + 3 * npl * m->nen) * elem;
  if (m->tan_work_bytes >= bytes) return FE_OK;
  if (m->lean) return FE_ERR_OOM;
  if (bytes > TAN_WORK_SMALL) {
    size_t free_b = 0, total_b = 0;
    FE_CUDA(cudaMemGetInfo(&free_b, &total_b));
    if (bytes > (free_b + m->tan_work_bytes) / 4) return FE_ERR_OOM;
  }
  if (m->tan_work) {
    FE_CUDA(cudaFreeAsync(m->tan_work, m->stream));
    m->device_bytes -= (int64_t)m->tan_work_bytes;
    m->tan_work = nullptr;
    m->tan_work_bytes = 0;
  }
  FE_TRY(fe_alloc_once(m, &m->tan_work, bytes));
  m->tan_work_bytes = bytes;
  return FE_OK;
}

template <int ORDER, class T>
static int launch_tangent_blocks(fe_mesh m, const double* d, T* K, T* B) {
  using C = Blk64Cfg<ORDER>;
  const double mass = m->dyn ? m->mass_c : 0.0, nen = C::NEN;
  const int npl = m->pres == 0 ? 0 : (m->pres == 2 ? 1 : 4);
  T *Ke = (T*)m->tan_work, *Be = Ke + (size_t)m->ne * C::NPAIR * 9;
  {
    FE_SCOPE(m, FE_PROF_TANGENT, (double)m->ne * (4 * nen + 84 + 24 * nen + sizeof(T) * (9.0 * C::NPAIR + 3.0 * npl * nen)));
    if constexpr (sizeof(T) == 8) {
      const int smem = (int)sizeof(T) * C::EB * C::NQ * (C::MS + (m->pres ? 12 : 0));
      FE_TRY(fe_kernel_smem((const void*)k_elem_blocks64<ORDER, T>, smem));
      k_elem_blocks64<ORDER, T><<<(m->ne + C::EB - 1) / C::EB, C::THREADS, smem, m->stream>>>(
          m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib, mass, Ke, Be);
    } else {
      using F = Blk32Cfg<ORDER>;
      const int smem = (int)sizeof(T) * F::EB * (F::PER_E + (m->pres ? F::NQ * 9 : 0));
      FE_TRY(fe_kernel_smem((const void*)k_elem_blocks32<ORDER>, smem));
      k_elem_blocks32<ORDER><<<(m->ne + F::EB - 1) / F::EB, F::THREADS, smem, m->stream>>>(
          m->ne, m->conn, m->geo, d, m->nn, m->pres, m->mp, m->fib, mass, Ke, Be);
    }
    FE_CUDA(cudaGetLastError());
  }
  FE_SCOPE(m, FE_PROF_TANGENT, (double)m->ne * (sizeof(T) * (9.0 * C::NPAIR + 3.0 * npl * nen) + 4 * nen * nen) +
                                   (double)m->nnzb * (9 * sizeof(T) + 4) + 12.0 * m->nn + 3.0 * sizeof(T) * m->nnz_up);
  k_gather_tangent<ORDER, T><<<(m->nn + TG_WARPS - 1) / TG_WARPS, 32 * TG_WARPS, 0, m->stream>>>(
      m->nn, m->node_ptr, m->color_list, m->emap, Ke, m->row_ptr, m->col, m->fixmask, K, npl, m->upmap, Be, m->up_ptr,
      B, m->nnzb);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

template <int ORDER, class T>
static int launch_tangent(fe_mesh m, const double* d, T* K, T* B) {
  using C = TanCfg<ORDER, T>;
  size_t smem = sizeof(T) * C::EPB * C::PER_E;
  const size_t nval = kv_count(m->nnzb);
  const int rc = tangent_workspace(m, sizeof(T));
  if (rc == FE_OK) return launch_tangent_blocks<ORDER, T>(m, d, K, B);
  if (rc != FE_ERR_OOM) return rc;
  FE_CUDA(cudaMemsetAsync(K, 0, nval * sizeof(T), m->stream));
  if (m->pres) FE_CUDA(cudaMemsetAsync(B, 0, (size_t)std::max<int64_t>(m->nnz_up, 1) * 3 * sizeof(T), m->stream));
  FE_TRY(fe_kernel_smem((const void*)k_elem_tangent<ORDER, T>, (int)smem));
  for (int c = 0; c < m->ncolors; c++) {
    int start = m->h_color_start[c], nel = m->h_color_start[c + 1] - start;
    if (nel == 0) continue;
    int grid = (nel + C::EPB - 1) / C::EPB;
    const double nen = C::NEN;
    FE_SCOPE(m, FE_PROF_TANGENT, (double)nel * (4 * nen + 84 + 4 + 24 * nen + 4 * nen * nen + nen +
                                                2.0 * 9 * sizeof(T) * nen * nen + (m->pres ? 16.0 * nen * 4 * sizeof(T) : 0)));
    k_elem_tangent<ORDER, T><<<grid, 256, smem, m->stream>>>(nel, m->perm + start, m->conn, m->geo, d, m->nn,
                                                             m->pres, m->mp, m->fib, m->emap, m->upmap,
                                                             m->fixmask, m->dyn ? m->mass_c : 0.0, K, B,
                                                             m->nnzb);
    FE_CUDA(cudaGetLastError());
  }
  return FE_OK;
}

// the tiled values; the last tile's padding is zero (every assembly writes the
// blocks)
template <class T>
static int alloc_values(fe_mesh m, T** K) {
  const size_t nval = kv_count(m->nnzb);
  FE_TRY(fe_alloc_t(m, K, nval));
  FE_CUDA(cudaMemsetAsync(*K, 0, nval * sizeof(T), m->stream));
  return FE_OK;
}

template <class T>
static int add_face_blocks(fe_mesh m, const double* d, T* K) {
  FE_SCOPE(m, FE_PROF_TANGENT, (double)m->nnz_ks * (4 + 4 + 72 + 2 * 9 * sizeof(T)));
  auto kern = m->order == 1 ? k_add_face_blocks<1, T> : k_add_face_blocks<2, T>;
  kern<<<(unsigned)((m->nnz_ks + 127) / 128), 128, 0, m->stream>>>(m->nnz_ks, m->ks_row, m->ks_col, m->ks_val,
                                                                   m->ks_kpos, m->fixmask, follower_faces(m), d,
                                                                   m->load, K);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

int fe_tangent_dev(fe_mesh m, const double* d, int precision) {
  if (precision < 0 || precision > 2) return fe_set_error("bad precision %d", precision), FE_ERR_ARG;
  if (precision == FE_PREC_MIXED_BF16 && m->pres)
    return fe_set_error("BF16 tangent storage is offered for the displacement form only"), FE_ERR_ARG;
  const size_t nval = kv_count(m->nnzb);  // tiles of 32 blocks (the last one zero-padded)
  const size_t nb = (size_t)(m->nnz_up > 0 ? m->nnz_up : 1) * 3;
  if (precision == FE_PREC_FP64) {
    if (!m->K64) FE_TRY(alloc_values(m, &m->K64));
    if (!m->Dinv64) FE_TRY(fe_alloc_t(m, &m->Dinv64, (size_t)m->nn * 9));
    if (m->pres && !m->B64) FE_TRY(fe_alloc_t(m, &m->B64, nb));
    if (m->order == 1) FE_TRY((launch_tangent<1, double>(m, d, m->K64, m->B64)));
    else FE_TRY((launch_tangent<2, double>(m, d, m->K64, m->B64)));
    if (m->nnz_ks) FE_TRY(add_face_blocks(m, d, m->K64));
    FE_SCOPE(m, FE_PROF_TANGENT, (double)m->nn * (4 + 1 + 72 + 72 + 72));
    k_diag_inverse<double, double><<<(m->nn + 255) / 256, 256, 0, m->stream>>>(m->nn, m->diag_pos, m->fixmask,
                                                                               m->K64, m->Dinv64);
  } else {
    if (!m->K32) FE_TRY(alloc_values(m, &m->K32));
    if (!m->Dinv32) FE_TRY(fe_alloc_t(m, &m->Dinv32, (size_t)m->nn * 9));
    if (m->pres && !m->B32) FE_TRY(fe_alloc_t(m, &m->B32, nb));
    if (m->order == 1) FE_TRY((launch_tangent<1, float>(m, d, m->K32, m->B32)));
    else FE_TRY((launch_tangent<2, float>(m, d, m->K32, m->B32)));
    if (m->nnz_ks) FE_TRY(add_face_blocks(m, d, m->K32));
    {
      FE_SCOPE(m, FE_PROF_TANGENT, (double)m->nn * (4 + 1 + 36 + 36 + 36));
      k_diag_inverse<float, float><<<(m->nn + 255) / 256, 256, 0, m->stream>>>(m->nn, m->diag_pos, m->fixmask,
                                                                             m->K32, m->Dinv32);
    }
    if (precision == FE_PREC_MIXED_BF16) {
      if (!m->K16) FE_TRY(fe_alloc_t(m, &m->K16, nval));
      FE_SCOPE(m, FE_PROF_TANGENT, 6.0 * nval);
      k_to_bf16<<<(unsigned)((nval + 255) / 256), 256, 0, m->stream>>>((int64_t)nval, m->K32, m->K16);
    }
  }
  FE_CUDA(cudaGetLastError());
  if (m->pres) {
    if (!m->Sd) FE_TRY(fe_alloc_t(m, &m->Sd, (size_t)m->np));
    FE_SCOPE(m, FE_PROF_TANGENT, (double)m->nnz_up * (8 + 3.0 * (precision == FE_PREC_FP64 ? 8 : 4) + 4) + 12.0 * m->np);
    if (precision == FE_PREC_FP64)
      k_schur_diag<double><<<(m->np + 7) / 8, 256, 0, m->stream>>>(m->np, m->pu_ptr, m->pu_col, m->pu_src,
                                                                       m->diag_pos, m->K64, m->B64, m->Sd);
    else
      k_schur_diag<float><<<(m->np + 7) / 8, 256, 0, m->stream>>>(m->np, m->pu_ptr, m->pu_col, m->pu_src,
                                                                      m->diag_pos, m->K32, m->B32, m->Sd);
    FE_CUDA(cudaGetLastError());
  }
  m->prec = precision;
  if (m->pc_type == 2 && precision == FE_PREC_MIXED_FP32) {  // BF16 fine level for the V-cycle's smoother
    const size_t nval = kv_count(m->nnzb);
    if (!m->K16) FE_TRY(fe_alloc_t(m, &m->K16, nval));
    FE_SCOPE(m, FE_PROF_TANGENT, 6.0 * nval);
    k_to_bf16<<<(unsigned)((nval + 255) / 256), 256, 0, m->stream>>>((int64_t)nval, m->K32, m->K16);
    FE_CUDA(cudaGetLastError());
  }
  if (m->pc_type >= 1) FE_TRY(fe_amg_setup(m));  // the AMG hierarchy of this tangent
  return FE_OK;
}

// ---------------------------------------------------------------- C ABI
extern "C" int fe_assemble_residual(fe_mesh m, const double* d, double* r, double* norm_out) {
  if (!m || !d || !r) return fe_set_error("NULL argument"), FE_ERR_ARG;
  FE_CUDA(cudaSetDevice(m->device));
  FE_TRY(fe_residual_dev(m, d, r, norm_out != nullptr));
  if (norm_out) {
    FE_CUDA(cudaMemcpyAsync(m->h_scal, m->scal, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  }
  FE_TRY(fe_check_device_error(m));
  if (norm_out) *norm_out = sqrt(m->h_scal[0]);
  return FE_OK;
}

extern "C" int fe_energy(fe_mesh m, const double* d, double* pi_out) {
  if (!m || !d || !pi_out) return fe_set_error("NULL argument"), FE_ERR_ARG;
  FE_CUDA(cudaSetDevice(m->device));
  FE_TRY(fe_energy_dev(m, d, pi_out));
  return fe_check_device_error(m);
}

extern "C" int fe_assemble_tangent(fe_mesh m, const double* d, int precision) {
  if (!m || !d) return fe_set_error("NULL argument"), FE_ERR_ARG;
  FE_CUDA(cudaSetDevice(m->device));
  FE_TRY(fe_tangent_dev(m, d, precision));
  return fe_check_device_error(m);
}

__global__ void k_widen(int64_t n, const float* __restrict__ s, double* __restrict__ d) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = (double)s[i];
}
__global__ void k_widen_bf(int64_t n, const __nv_bfloat16* __restrict__ s, double* __restrict__ d) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = (double)__bfloat162float(s[i]);
}

static int copy_out(fe_mesh m, double* host, const double* d64, const float* d32, const __nv_bfloat16* d16,
                    int64_t n) {
  if (!host) return FE_OK;
  if (d64) {
    FE_CUDA(cudaMemcpy(host, d64, n * sizeof(double), cudaMemcpyDeviceToHost));
    return FE_OK;
  }
  double* tmp = nullptr;
  FE_TRY(fe_alloc_t(m, &tmp, (size_t)n));
  m->device_bytes -= n * (int64_t)sizeof(double);  // (freed below)
  if (d16) k_widen_bf<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(n, d16, tmp);
  else k_widen<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(n, d32, tmp);
  cudaError_t e = cudaStreamSynchronize(m->stream);
  if (e == cudaSuccess) e = cudaMemcpy(host, tmp, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFreeAsync(tmp, m->stream);
  cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return fe_set_error("%s", cudaGetErrorString(e)), FE_ERR_CUDA;
  return FE_OK;
}

extern "C" int fe_tangent_copy(fe_mesh m, double* val, double* bup, double* dinv) {
  if (!m) return fe_set_error("NULL mesh"), FE_ERR_ARG;
  if (m->prec < 0) return fe_set_error("no tangent assembled"), FE_ERR_STATE;
  FE_CUDA(cudaSetDevice(m->device));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  bool f64 = m->prec == FE_PREC_FP64;
  bool b16 = m->prec == FE_PREC_MIXED_BF16;
  if (val) {  // device values are tiled (kv_index); the copy is block-major [nnzb][3][3]
    std::vector<double> tv(kv_count(m->nnzb));
    FE_TRY(copy_out(m, tv.data(), f64 ? m->K64 : nullptr, f64 ? nullptr : m->K32, b16 ? m->K16 : nullptr,
                    (int64_t)tv.size()));
    for (int64_t p = 0; p < m->nnzb; p++)
      for (int c = 0; c < 9; c++) val[p * 9 + c] = tv[kv_index(p, c)];
  }
  if (m->pres) FE_TRY(copy_out(m, bup, f64 ? m->B64 : nullptr, f64 ? nullptr : m->B32, nullptr, m->nnz_up * 3));
  FE_TRY(copy_out(m, dinv, f64 ? m->Dinv64 : nullptr, f64 ? nullptr : m->Dinv32, nullptr, (int64_t)m->nn * 9));
  return FE_OK;
}

// ---------------------------------------------------------------- elastodynamics
// Newmark average acceleration (beta = 1/4, gamma = 1/2): the state d_n,
// v_n, a_n gives the predictors dhat = d_n + dt v_n + dt^2/4 a_n and
// dtil = d_n + dt/2 v_n; the step's residual is R(d) + 4/dt^2 M (d - dhat)
// + 2/dt C (d - dtil).  Layout of m->dyn: [6][3 nn] d_n, v_n, a_n, dhat,
// dtil, fdyn.

int fe_upload_face_values(fe_mesh m) {
  const size_t n = m->h_ks_spring.size();
  std::vector<double> v(m->h_ks_spring);
  if (m->dyn && m->has_dashpots)
    for (size_t i = 0; i < n; i++) v[i] += 2.0 / m->dyn_dt * m->h_ks_dashpot[i];
  if (!m->ks_val) FE_TRY(fe_alloc_t(m, &m->ks_val, n ? n : 1));
  if (n) FE_CUDA(cudaMemcpyAsync(m->ks_val, v.data(), n * sizeof(double), cudaMemcpyHostToDevice, m->stream));
  if (m->has_dashpots && !m->kc_val) {
    FE_TRY(fe_alloc_t(m, &m->kc_val, n));
    FE_CUDA(cudaMemcpyAsync(m->kc_val, m->h_ks_dashpot.data(), n * sizeof(double), cudaMemcpyHostToDevice,
                            m->stream));
  }
  FE_CUDA(cudaStreamSynchronize(m->stream));  // v is a host temporary
  return FE_OK;
}

// mode 0 (set): the state from d, v, a (nullptr: zero); mode 1 (advance):
// a = 4/dt^2 (d - dhat), v = 2/dt (d - dtil) from the converged d, then d_n = d.
// Either way the predictors of the next step follow.
__global__ void k_newmark_state(int64_t n3, int mode, double dt, const double* __restrict__ d,
                                const double* __restrict__ v, const double* __restrict__ a,
                                double* __restrict__ st) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  double* dn = st;
  double* vn = st + n3;
  double* an = st + 2 * n3;
  double* dhat = st + 3 * n3;
  double* dtil = st + 4 * n3;
  double di, vi, ai;
  if (mode == 0) {
    di = d ? d[i] : 0.0;
    vi = v ? v[i] : 0.0;
    ai = a ? a[i] : 0.0;
  } else {
    di = d[i];
    ai = 4.0 / (dt * dt) * (di - dhat[i]);
    vi = 2.0 / dt * (di - dtil[i]);
  }
  dn[i] = di;
  vn[i] = vi;
  an[i] = ai;
  dhat[i] = di + dt * vi + 0.25 * dt * dt * ai;
  dtil[i] = di + 0.5 * dt * vi;
}

// fdyn = mass_c M dhat + 2/dt C dtil per node (M gathered from the
// elements of the node in node_list order, C from the face pattern) and the
// constant of the step functional, (mass_c dhat.M dhat + 2/dt dtil.C dtil) / 2
template <int ORDER>
__global__ void __launch_bounds__(256) k_newmark_load(int nn, const int* __restrict__ node_ptr,
                                                      const int* __restrict__ node_list, const int* __restrict__ conn,
                                                      const double* __restrict__ geo, double mass_c, double cc,
                                                      const int* __restrict__ ks_ptr, const int* __restrict__ ks_col,
                                                      const double* __restrict__ kc_val, double* __restrict__ st,
                                                      double* red, unsigned* ticket, double* out) {
  constexpr int NEN = ORDER == 1 ? 4 : 10;
  const int64_t n3 = 3 * (int64_t)nn;
  const double* dhat = st + 3 * n3;
  const double* dtil = st + 4 * n3;
  double* fdyn = st + 5 * n3;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  double acc = 0.0;
  if (t < nn) {
    double mh[3] = {0.0, 0.0, 0.0}, ch[3] = {0.0, 0.0, 0.0};
    for (int k = node_ptr[t]; k < node_ptr[t + 1]; k++) {
      const int slot = node_list[k], e = slot / NEN, a = slot % NEN;
      const double vol = geo[(size_t)e * 10 + 9];
      const int* c = conn + (size_t)e * NEN;
      for (int b = 0; b < NEN; b++) {
        const double w = vol * mass_hat(ORDER, a, b);
        const double* u = dhat + 3 * (size_t)c[b];
        for (int i = 0; i < 3; i++) mh[i] += w * u[i];
      }
    }
    if (kc_val)
      for (int k = ks_ptr[t]; k < ks_ptr[t + 1]; k++) {
        const double* kv = kc_val + (size_t)k * 9;
        const double* u = dtil + 3 * (size_t)ks_col[k];
        for (int i = 0; i < 3; i++) ch[i] += kv[3 * i] * u[0] + kv[3 * i + 1] * u[1] + kv[3 * i + 2] * u[2];
      }
    for (int i = 0; i < 3; i++) {
      fdyn[3 * (size_t)t + i] = mass_c * mh[i] + cc * ch[i];
      acc += 0.5 * (mass_c * dhat[3 * (size_t)t + i] * mh[i] + cc * dtil[3 * (size_t)t + i] * ch[i]);
    }
  }
  grid_sum_finish(acc, red, ticket, out);
}

static int newmark_update(fe_mesh m, int mode, const double* d, const double* v, const double* a) {
  const int64_t n3 = 3 * (int64_t)m->nn;
  const int grid = (m->nn + 255) / 256;
  if (grid > RED_SLOTS) return fe_set_error("mesh too large for the reduction buffer"), FE_ERR_ARG;
  {
    FE_SCOPE(m, FE_PROF_OTHER, (mode == 0 ? 3.0 : 1.0) * 8 * n3 + (mode == 0 ? 0.0 : 16.0 * n3) + 40.0 * n3);
    k_newmark_state<<<(unsigned)((n3 + 255) / 256), 256, 0, m->stream>>>(n3, mode, m->dyn_dt, d, v, a, m->dyn);
  }
  FE_CUDA(cudaGetLastError());
  {
    FE_SCOPE(m, FE_PROF_OTHER, (double)m->ne * m->nen * (8.0 + 4.0 * m->nen + 24.0 * m->nen) + 72.0 * m->nnz_ks);
    auto kern = m->order == 1 ? k_newmark_load<1> : k_newmark_load<2>;
    kern<<<grid, 256, 0, m->stream>>>(m->nn, m->node_ptr, m->node_list, m->conn, m->geo, m->mass_c,
                                      2.0 / m->dyn_dt, m->ks_ptr, m->ks_col, m->kc_val, m->dyn, m->red,
                                      m->red_ticket, m->scal + 40);
  }
  FE_CUDA(cudaGetLastError());
  FE_CUDA(cudaMemcpyAsync(m->h_scal + 40, m->scal + 40, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  FE_TRY(fe_check_device_error(m));
  m->dyn_const = m->h_scal[40];
  return FE_OK;
}

extern "C" int fe_set_dynamics(fe_mesh m, double rho, double dt) {
  if (!m) return fe_set_error("NULL mesh"), FE_ERR_ARG;
  if (!std::isfinite(rho) || !std::isfinite(dt)) return fe_set_error("rho and dt must be finite"), FE_ERR_ARG;
  FE_CUDA(cudaSetDevice(m->device));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  if (rho <= 0.0 || dt <= 0.0) {  // static again; the state storage stays allocated
    const bool was = m->dyn != nullptr;
    m->dyn_rho = m->dyn_dt = m->mass_c = m->dyn_const = 0.0;
    if (was) {
      double* keep = m->dyn;
      m->dyn = nullptr;
      FE_TRY(fe_upload_face_values(m));
      m->dyn_keep = keep;
    }
    return FE_OK;
  }
  if (!m->dyn) {
    if (!m->dyn_keep) FE_TRY(fe_alloc_t(m, &m->dyn_keep, 6 * 3 * (size_t)m->nn));
    m->dyn = m->dyn_keep;
  }
  m->dyn_rho = rho;
  m->dyn_dt = dt;
  m->mass_c = 4.0 * rho / (dt * dt);
  FE_TRY(fe_upload_face_values(m));
  return newmark_update(m, 0, nullptr, nullptr, nullptr);
}

extern "C" int fe_dynamics_set(fe_mesh m, const double* d, const double* v, const double* a) {
  if (!m) return fe_set_error("NULL mesh"), FE_ERR_ARG;
  if (!m->dyn) return fe_set_error("dynamics is off (fe_set_dynamics)"), FE_ERR_STATE;
  FE_CUDA(cudaSetDevice(m->device));
  return newmark_update(m, 0, d, v, a);
}

extern "C" int fe_dynamics_advance(fe_mesh m, const double* d) {
  if (!m || !d) return fe_set_error("NULL argument"), FE_ERR_ARG;
  if (!m->dyn) return fe_set_error("dynamics is off (fe_set_dynamics)"), FE_ERR_STATE;
  FE_CUDA(cudaSetDevice(m->device));
  return newmark_update(m, 1, d, nullptr, nullptr);
}

extern "C" int fe_dynamics_get(fe_mesh m, double* v, double* a) {
  if (!m) return fe_set_error("NULL mesh"), FE_ERR_ARG;
  if (!m->dyn) return fe_set_error("dynamics is off (fe_set_dynamics)"), FE_ERR_STATE;
  FE_CUDA(cudaSetDevice(m->device));
  const size_t n3 = 3 * (size_t)m->nn;
  if (v) FE_CUDA(cudaMemcpyAsync(v, m->dyn + n3, n3 * sizeof(double), cudaMemcpyDeviceToDevice, m->stream));
  if (a) FE_CUDA(cudaMemcpyAsync(a, m->dyn + 2 * n3, n3 * sizeof(double), cudaMemcpyDeviceToDevice, m->stream));
  return fe_check_device_error(m);
}

FE_DBG_BOUNDS_READER(fe_dbg_bounds_assemble)
