// fe_batch.cu -- many small nonlinear solves in one launch (the kernel is in
// fe_batch_kernel.cuh): the requests' tables, workspace and launch.
#include <cstring>

#include "fe_batch_kernel.cuh"

// ---------------------------------------------------------------- host side
static size_t batch_smem(int order, int prec, int restart) {
  const size_t tan = order == 1 ? (prec == FE_PREC_FP64 ? sizeof(double) * TanCfg<1, double>::EPB * TanCfg<1, double>::PER_E
                                                       : sizeof(float) * TanCfg<1, float>::EPB * TanCfg<1, float>::PER_E)
                                : (prec == FE_PREC_FP64 ? sizeof(double) * TanCfg<2, double>::EPB * TanCfg<2, double>::PER_E
                                                       : sizeof(float) * TanCfg<2, float>::EPB * TanCfg<2, float>::PER_E);
  const size_t gm = sizeof(double) * ((size_t)(restart + 1) * restart + 4 * (size_t)restart + 1 +
                                      2 * VLANES / 32 * 8 + (size_t)(restart / 8 + 1) * BATCH_GRAM);
  return (tan + 15) / 16 * 16 + gm;
}

const void* fe_batch_kernel_p1(bool f64, int nt) { return batch_kernel<1>(f64, nt); }

static const void* pick_kernel(int order, int prec, int nt) {
  return order == 1 ? fe_batch_kernel_p1(prec == FE_PREC_FP64, nt) : fe_batch_kernel_p2(prec == FE_PREC_FP64, nt);
}

extern "C" int fe_batch_supported(fe_mesh m, int method, const nl_opts* o) {
  if (!m) return 0;
  if (m->pres || m->nff || m->dyn || m->ncolors > BATCH_MAX_COLORS) return 0;
  if (method < NL_NK || method > NL_IB) return 0;
  if (o && (o->pc_type != 0 || o->precision == FE_PREC_MIXED_BF16 || o->jac_lag > 1 || o->hess_reassemble > 0 ||
            o->ib_adaptive))
    return 0;
  // the Hessenberg matrix lives in shared memory: GMRES(m) with m <= BATCH_MAX_RESTART
  if (!o || o->ksp_restart <= 0 || o->ksp_restart > BATCH_MAX_RESTART) return 0;
  if ((method == NL_B || method == NL_IB) && o && o->lbfgs_m > BATCH_HIST) return 0;
  return 1;
}

// workspace of one request (device), allocated per batch call
struct BatchWork {
  double* base = nullptr;
  void* K = nullptr;
  void* Dinv = nullptr;
};

// one launch for requests of one order and one precision
static int batch_group(int nreq, fe_mesh* meshes, const int* methods, const double* tols, const int* max_its,
                       const nl_opts* opts, double** d, int threads, fe_batch_out* out_host) {
  const fe_mesh m0 = meshes[0];
  const int order = m0->order;
  const int prec = opts[0].precision;
  std::vector<BatchReq> h(nreq);
  std::vector<void*> allocs;
  cudaStream_t stream = m0->stream;
  // stream-ordered allocations: no device-wide synchronisation, so batches
  // on other streams keep running
  auto cleanup = [&]() {
    for (void* p : allocs) cudaFreeAsync(p, stream);
  };
  std::vector<size_t> off_base(nreq), off_K(nreq), off_D(nreq);
  size_t total = 0;
  auto take = [&](size_t bytes) {
    const size_t o = total;
    total += (bytes + 255) / 256 * 256;
    return o;
  };
  int restart_max = 1;
  for (int i = 0; i < nreq; i++) {
    fe_mesh m = meshes[i];
    nl_opts o;
    nl_opts_default((nl_method)methods[i], &o);
    if (opts) {
      const nl_opts& u = opts[i];
      o.precision = u.precision;
      if (u.ksp_rtol >= 0) o.ksp_rtol = u.ksp_rtol;
      if (u.ksp_atol >= 0) o.ksp_atol = u.ksp_atol;
      if (u.ew_rtol0 > 0) o.ew_rtol0 = u.ew_rtol0;
      if (u.ew_rtolmax > 0) o.ew_rtolmax = u.ew_rtolmax;
      if (u.ksp_restart > 0) o.ksp_restart = u.ksp_restart;
      if (u.ksp_max_it > 0) o.ksp_max_it = u.ksp_max_it;
      if (u.lbfgs_m > 0) o.lbfgs_m = u.lbfgs_m;
      if (u.dtol > 0) o.dtol = u.dtol;
      o.apply_dirichlet = u.apply_dirichlet;
    }
    if (m->order != order || o.precision != prec) {
      cleanup();
      return fe_set_error("internal: a launch group needs one order and one precision"), FE_ERR_ARG;
    }
    restart_max = std::max(restart_max, o.ksp_restart);
    BatchReq& q = h[i];
    std::memset(&q, 0, sizeof(q));
    q.nn = m->nn;
    q.ne = m->ne;
    q.ncolors = m->ncolors;
    q.nnzb = m->nnzb;
    q.conn = m->conn;
    q.perm = m->perm;
    q.node_ptr = m->node_ptr;
    q.node_list = m->node_list;
    q.row_ptr = m->row_ptr;
    q.col = m->col;
    q.emap = m->emap;
    q.diag_pos = m->diag_pos;
    q.ks_ptr = m->ks_ptr;
    q.ks_col = m->ks_col;
    q.ks_kpos = m->ks_kpos;
    q.geo = m->geo;
    q.X = m->X;
    q.fib = m->fib;
    q.fext1 = m->fext1;
    q.ks_val = m->ks_val;
    q.fixmask = m->fixmask;
    q.mp = m->mp;
    q.load = m->load;
    for (int c = 0; c <= m->ncolors; c++) q.cstart[c] = m->h_color_start[c];
    q.method = methods[i];
    q.max_it = max_its[i];
    q.restart = o.ksp_restart;
    q.kmaxit = o.ksp_max_it;
    q.mcap = o.lbfgs_m;
    q.tol = tols[i];
    q.ksp_rtol = o.ksp_rtol;
    q.ksp_atol = o.ksp_atol;
    q.ew0 = o.ew_rtol0;
    q.ewmax = o.ew_rtolmax;
    q.dtol = o.dtol;
    const int64_t n = 3 * (int64_t)m->nn;
    const int64_t nvec = 7 + (q.restart + 1) + ((q.method >= NL_B) ? 2 * (int64_t)std::min(q.mcap, BATCH_HIST) : 0);
    const int64_t nrel = (int64_t)m->ne * m->nen * 3;
    const size_t sval = prec == FE_PREC_FP64 ? 8 : 4;
    off_base[i] = take(sizeof(double) * (size_t)(nvec * n + nrel));
    off_K[i] = take(sval * kv_count(m->nnzb));
    off_D[i] = take(sval * 9 * (size_t)m->nn);
  }
  FE_CUDA(cudaSetDevice(m0->device));
  char* pool = nullptr;
  if (cudaMallocAsync((void**)&pool, total, stream) != cudaSuccess)
    return fe_set_error("batch workspace allocation failed"), FE_ERR_OOM;
  allocs.push_back(pool);
  for (int i = 0; i < nreq; i++) {
    BatchReq& q = h[i];
    const int64_t n = 3 * (int64_t)meshes[i]->nn;
    const int64_t nrel = (int64_t)meshes[i]->ne * meshes[i]->nen * 3;
    double* base = (double*)(pool + off_base[i]);
    q.d = d[i];
    q.r = base;
    q.rn = base + n;
    q.dl = base + 2 * n;
    q.t = base + 3 * n;
    q.w = base + 4 * n;
    q.zb = base + 5 * n;
    q.gr = base + 6 * n;
    q.rel = base + 7 * n;
    q.V = q.rel + nrel;
    q.S = q.V + (int64_t)(q.restart + 1) * n;
    q.Y = q.S + (int64_t)std::min(q.mcap, BATCH_HIST) * n;
    q.K = pool + off_K[i];
    q.Dinv = pool + off_D[i];
  }
  BatchReq* dq = nullptr;
  fe_batch_out* dout = nullptr;
  if (cudaMallocAsync((void**)&dq, sizeof(BatchReq) * nreq, stream) != cudaSuccess) {
    cleanup();
    return fe_set_error("batch table allocation failed"), FE_ERR_OOM;
  }
  allocs.push_back(dq);
  if (cudaMallocAsync((void**)&dout, sizeof(fe_batch_out) * nreq, stream) != cudaSuccess) {
    cleanup();
    return fe_set_error("batch table allocation failed"), FE_ERR_OOM;
  }
  allocs.push_back(dout);
  for (int i = 0; i < nreq; i++) h[i].out = dout + i;
  // Dirichlet values of each request's load first (on each mesh's stream),
  // then the batch on the first mesh's stream
  for (int i = 0; i < nreq; i++) {
    if (!opts || opts[i].apply_dirichlet) {
      int rc = fe_apply_dirichlet(meshes[i], d[i]);
      if (rc != FE_OK) {
        cleanup();
        return rc;
      }
    }
    if (meshes[i]->stream != stream) {
      cudaError_t e = cudaStreamSynchronize(meshes[i]->stream);
      if (e != cudaSuccess) {
        cleanup();
        return fe_set_error("%s", cudaGetErrorString(e)), FE_ERR_CUDA;
      }
    }
  }
  cudaError_t e = cudaMemcpyAsync(dq, h.data(), sizeof(BatchReq) * nreq, cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(dout, 0, sizeof(fe_batch_out) * nreq, stream);
  const size_t smem = batch_smem(order, prec, restart_max);
  const void* fn = pick_kernel(order, prec, threads);
  if (e == cudaSuccess && fe_kernel_smem(fn, (int)smem) != FE_OK) {
    cleanup();
    return FE_ERR_CUDA;
  }
  if (e == cudaSuccess) {
    void* args[] = {(void*)&dq};
    e = cudaLaunchKernel(fn, dim3(nreq), dim3(threads), args, smem, stream);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(out_host, dout, sizeof(fe_batch_out) * nreq, cudaMemcpyDeviceToHost, stream);
  cleanup();  // stream-ordered: after the kernel and the copy-back
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return fe_set_error("batch solve: %s", cudaGetErrorString(e)), FE_ERR_CUDA;
  return FE_OK;
}

extern "C" int fe_batch_solve(int nreq, fe_mesh* meshes, const int* methods, const double* tols,
                              const int* max_its, const nl_opts* opts, double** d, int threads,
                              fe_batch_out* out_host) {
  if (nreq <= 0) return FE_OK;
  if (!meshes || !methods || !tols || !max_its || !opts || !d || !out_host)
    return fe_set_error("NULL argument"), FE_ERR_ARG;
  if (threads != 128 && threads != 256) return fe_set_error("threads must be 128 or 256"), FE_ERR_ARG;
  for (int i = 0; i < nreq; i++) {
    if (!meshes[i] || !d[i]) return fe_set_error("NULL mesh or vector of request %d", i), FE_ERR_ARG;
    if (meshes[i]->device != meshes[0]->device) return fe_set_error("a batch runs on one device"), FE_ERR_ARG;
    if (!fe_batch_supported(meshes[i], methods[i], &opts[i]))
      return fe_set_error("request %d is not supported by the batched solver", i), FE_ERR_ARG;
  }
  // one launch per (order, precision), in order of first appearance
  std::vector<int> done(nreq, 0);
  for (int i0 = 0; i0 < nreq; i0++) {
    if (done[i0]) continue;
    std::vector<int> idx;
    for (int i = i0; i < nreq; i++)
      if (!done[i] && meshes[i]->order == meshes[i0]->order && opts[i].precision == opts[i0].precision) {
        idx.push_back(i);
        done[i] = 1;
      }
    const size_t g = idx.size();
    std::vector<fe_mesh> gm(g);
    std::vector<int> gmeth(g), gmax(g);
    std::vector<double> gtol(g);
    std::vector<nl_opts> gopt(g);
    std::vector<double*> gd(g);
    std::vector<fe_batch_out> gout(g);
    for (size_t k = 0; k < g; k++) {
      gm[k] = meshes[idx[k]];
      gmeth[k] = methods[idx[k]];
      gmax[k] = max_its[idx[k]];
      gtol[k] = tols[idx[k]];
      gopt[k] = opts[idx[k]];
      gd[k] = d[idx[k]];
    }
    FE_TRY(batch_group((int)g, gm.data(), gmeth.data(), gtol.data(), gmax.data(), gopt.data(), gd.data(), threads,
                       gout.data()));
    for (size_t k = 0; k < g; k++) out_host[idx[k]] = gout[k];
  }
  return FE_OK;
}

FE_DBG_BOUNDS_READER(fe_dbg_bounds_batch)
