"""Launch rules of the kernels at the sizes where they change: edges of
tiles, remainders and the smallest and largest sizes of each branch, against
the CPU oracle or against the general path."""
import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fe():
    import __graft_entry__ as g
    g.build()
    import paper_2203_05610_gb300 as fe
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return fe


# unknowns 150 (one block in both forms), 729 and 1,500 (several blocks only
# in the blocked form), 1,800 (several in both), 39,375 (a slice of 264 per
# SM), 151,290 (996 values: 256 threads x 4), 249,696 (1,644: the long-slice
# kernel)
@pytest.mark.parametrize("orthog", [0, 2])
@pytest.mark.parametrize("size", [(4, 4, 1), (8, 8, 2), (9, 9, 4), (9, 9, 5), (24, 24, 20), (40, 40, 29),
                                  (50, 50, 31)])
def test_arnoldi_launch_shapes(fe, size, orthog):
    # both sides run exactly 24 iterations in cycles of 13 (a full block of
    # eight basis vectors and a part of one); the projections are the same, so
    # the iterates differ by rounding (FP64 sums of n terms in another order:
    # below 1e-9 relative, the bound of the longer multi-block test)
    w = W.cook(*size, order=1, nu=0.3)
    m, om = fe.Mesh(w), O.Mesh(w)
    d = 0.02 * np.random.default_rng(3).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    dg = torch.from_numpy(d).cuda()
    om.tangent(d)
    m.tangent(dg)
    b = np.random.default_rng(4).standard_normal(om.ndof)
    x, it, res = om.gmres(b, rtol=1e-14, atol=0.0, restart=13, max_it=24)
    xg, itg, resg = m.gmres(torch.from_numpy(b).cuda(), rtol=1e-14, atol=0.0, restart=13, max_it=24, orthog=orthog)
    assert it == itg == 24
    assert abs(resg - res) <= 1e-8 * res, (resg, res)
    assert np.linalg.norm(xg.cpu().numpy() - x) <= 1e-9 * np.linalg.norm(x)


# block counts around one tile, one tile per warp of a wave (58k blocks in
# FP64, 117k in FP32) and beyond it, short P1 rows and long P2 rows
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed_fp32", 2e-5)])
@pytest.mark.parametrize("size,order", [((1, 1, 1), 1), ((2, 2, 1), 2), ((20, 20, 8), 1), ((22, 21, 9), 1),
                                        ((29, 27, 8), 1), ((30, 31, 9), 1), ((13, 11, 5), 2)])
def test_streamed_spmv_ranges(fe, size, order, precision, tol):
    # bounds of the parity tests: FP64 a few ulps of the largest entry, FP32
    # assembly and sums 2e-5 of it
    w = W.cook(*size, order=order, nu=0.3)
    m, om = fe.Mesh(w), O.Mesh(w)
    d = 0.02 * np.random.default_rng(5).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    om.tangent(d)
    m.tangent(torch.from_numpy(d).cuda(), precision)
    x = np.random.default_rng(6).standard_normal(om.ndof)
    y, yg = om.spmv(x), m.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.abs(yg - y).max() <= tol * np.abs(y).max()


# coarse rows of more than one chunk of the products (70 to 85 entries), the
# power steps in one launch (38 rows, 884 blocks) and in 15 (73 rows on)
@pytest.mark.parametrize("n", [4, 6, 8, 12])
def test_amg_setup_sizes(fe, n):
    # bounds of the hierarchy test: radii 1e-12, operators 1e-11, prolongators
    # 1e-12 of the largest entry; FP32 arithmetic 2e-5 per product of three
    # factors, 1e-4 for the sums of a row
    w = W.twist(n)
    m, om = fe.Mesh(w), O.Mesh(w)
    d = 0.002 * np.random.default_rng(7).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    dg = torch.from_numpy(d).cuda()
    om.set_pc("amg")
    om.tangent(d)
    m.set_pc("amg")
    x = np.random.default_rng(8).standard_normal(om.ndof)
    z = om.pc(x)
    for prec, tr, tv, tz in (("fp64", 1e-12, 1e-11, 1e-10), ("mixed_fp32", 1e-5, 1e-4, 2e-3)):
        m.tangent(dg, prec)
        ol, gl = om.amg_levels(), m.amg_levels()
        assert len(ol) == len(gl)
        for lv, (o, g) in enumerate(zip(ol, gl)):
            if lv < len(ol) - 1:
                assert abs(g["rho"] - o["rho"]) <= tr * o["rho"], lv
                assert np.abs(g["pval"] - o["pval"]).max() <= tv * np.abs(o["pval"]).max(), lv
            if lv > 0:
                assert np.array_equal(g["col"], o["col"])
                assert np.abs(g["val"] - o["val"]).max() <= tv * np.abs(o["val"]).max(), lv
        zg = m.pc(torch.from_numpy(x).cuda()).cpu().numpy()
        assert np.abs(zg - z).max() <= tz * np.abs(z).max(), prec


def _hub(order):
    """A vertex inside a ball of 33 points on a sphere (62 elements): its P2 row has 160 blocks."""
    from scipy.spatial import ConvexHull
    k = np.arange(33) + 0.5
    phi, th = np.arccos(1 - 2 * k / 33), np.pi * (1 + 5 ** 0.5) * k
    pts = np.stack([np.cos(th) * np.sin(phi), np.sin(th) * np.sin(phi), np.cos(phi)], axis=1)
    tri = ConvexHull(pts).simplices.astype(np.int64)
    flip = np.einsum("ij,ij->i", pts[tri[:, 0]], np.cross(pts[tri[:, 1]], pts[tri[:, 2]])) < 0
    tri[flip] = tri[flip][:, [0, 2, 1]]
    w = dict(W.cook(1, 1, 1, order=order, nu=0.3))
    w["coords"] = np.concatenate([np.zeros((1, 3)), pts])
    w["tets"] = np.concatenate([np.zeros((len(tri), 1), dtype=tri.dtype), tri + 1], axis=1).astype(w["tets"].dtype)
    w["dir_group"] = np.array([0, 1] + [0] * 32, dtype=w["dir_group"].dtype)
    w["faces"], w["face_kind"], w["face_data"] = w["faces"][:0], w["face_kind"][:0], w["face_data"][:0]
    return w


# 6 elements (less than a tile of 16 or 64), 96 (six tiles of 16), 144 and 150
# (a part tile), rows of one chunk of 96 blocks and of two
TANGENT = {"6": lambda o: W.cook(1, 1, 1, order=o, nu=0.3), "96": lambda o: W.cook(4, 2, 2, order=o, nu=0.3),
           "144": lambda o: W.cook(4, 3, 2, order=o, nu=0.3), "150": lambda o: W.cook(5, 5, 1, order=o, nu=0.3),
           "hub": _hub}


def _check_tangent(m, om, d, precision, tol):
    om.tangent(d)
    m.tangent(torch.from_numpy(d).cuda(), precision)
    x = np.random.default_rng(6).standard_normal(om.ndof)
    y = om.spmv(x)
    for _ in range(2):  # nothing of the first assembly stays in the second
        yg = m.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
        assert np.abs(yg - y).max() <= tol * np.abs(y).max()
        m.tangent(torch.from_numpy(d).cuda(), precision)


# bounds of the parity tests: FP64 1e-12, FP32 assembly and sums 2e-5 of the
# largest entry
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed_fp32", 2e-5)])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("case", list(TANGENT))
def test_tangent_tiles_and_rows(fe, case, order, precision, tol):
    w = TANGENT[case](order)
    m, om = fe.Mesh(w), O.Mesh(w)
    d = 0.01 * np.random.default_rng(9).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    _check_tangent(m, om, d, precision, tol)


def test_tangent_without_workspace(fe):
    # device memory that holds the matrix but not the element blocks (94 MB
    # and 128 MB, of 150 MB free): assembled colour by colour, to the same bounds
    w = W.cook(30, 30, 6, order=2, nu=0.3)
    m, om = fe.Mesh(w), O.Mesh(w)
    d = 0.01 * np.random.default_rng(9).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    torch.cuda.synchronize()
    hog = []
    while True:  # in pieces: the library's pool keeps what it has
        free = torch.cuda.mem_get_info()[0] - (150 << 20)
        if free < (2 << 20):
            break
        hog.append(torch.empty(min(free, 32 << 30), dtype=torch.uint8, device="cuda"))
    try:
        _check_tangent(m, om, d, "fp64", 1e-12)
    finally:
        del hog
        torch.cuda.empty_cache()


# element kernels of the residual: 6 and more P1 elements, P2 meshes on both sides
# of 6,080 elements, every law, statically and in a Newmark step
@pytest.mark.parametrize("case", ["cook1_6", "cook1_390", "cook2_6000", "cook2_6144", "twist_6000", "twist_7986",
                                  "heart1_12288"])
def test_residual_element_kernels(fe, case):
    # FP64 sums of a node's elements in the oracle's terms: a few ulps of the
    # largest contribution, 1e-12 of the largest entry as in the parity tests
    w = {"cook1_6": lambda: W.cook(1, 1, 1, order=1, nu=0.3), "cook1_390": lambda: W.cook(13, 5, 1, order=1, nu=0.3),
         "cook2_6000": lambda: W.cook(20, 10, 5, order=2, nu=0.3),
         "cook2_6144": lambda: W.cook(16, 16, 4, order=2, nu=0.49),
         "twist_6000": lambda: W.twist(10), "twist_7986": lambda: W.twist(11),
         "heart1_12288": lambda: W.heart(nr=2, nc=32, nl=32, order=1)}[case]()
    m, om = fe.Mesh(w), O.Mesh(w)
    m.set_load(0.4, 0.1)
    om.set_load(0.4, 0.1)
    d = 0.002 * np.random.default_rng(10).standard_normal(om.ndof)
    om.apply_dirichlet(d)
    dg = torch.from_numpy(d).cuda()
    r = om.residual(d)
    r = r[0] if isinstance(r, tuple) else r
    rg, norm = m.residual(dg)
    assert np.abs(rg.cpu().numpy() - r).max() <= 1e-12 * np.abs(r).max()
    assert abs(norm - np.linalg.norm(r)) <= 1e-12 * np.linalg.norm(r)
    if case.startswith("twist"):
        return
    for mesh in (m, om):
        mesh.set_dynamics(1e-3, 0.1)
    r = om.residual(d)
    r = r[0] if isinstance(r, tuple) else r
    rg, _ = m.residual(dg)
    assert np.abs(rg.cpu().numpy() - r).max() <= 1e-12 * np.abs(r).max()


# unknowns 225 to 1,989: one to eight values per lane of the batch kernel's
# orthogonalisation; 2,160: beyond it.  Cycles of 20 end in a part block.
@pytest.mark.parametrize("size", [(4, 4, 2), (5, 5, 2), (7, 7, 2), (8, 8, 3), (9, 9, 3), (10, 9, 3), (13, 12, 2),
                                  (16, 12, 2), (15, 14, 2)])
@pytest.mark.parametrize("restart", [20, 100])
def test_batch_orthogonalisation_sizes(fe, size, restart):
    # FP64 Newton with tight inner solves ends far below its tolerance, so the
    # solutions of both paths agree to the residual's 1e-10 times a condition
    # of 1e2: 1e-8; the CTA shapes agree bit for bit.  Iteration counts are
    # compared where the cycles hold the whole of the convergence (100 vectors
    # and up to 1,000 unknowns); short cycles stagnate, and rounding alone
    # moves their counts by a tenth.
    w = W.cook(*size, order=1, nu=0.3)
    opts = dict(ksp_restart=restart, ksp_rtol=1e-6, ksp_atol=0.0, precision="fp64")
    m = fe.Mesh(w)
    m.set_load(0.1)
    out = []
    for nt in (128, 256):
        d = m.zeros()
        st = fe.batch_solve([m], ["NK"], [d], [1e-10], opts=opts, threads=nt)[0]
        assert st["status"] == 0 and st["rfinal"] <= 1e-10 * st["r0"]
        out.append((d, st["lit_total"]))
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    d, st = m.solve("NK", m.zeros(), tol=1e-10, opts=opts)
    assert st["status"] == 0
    assert torch.linalg.norm(out[0][0] - d) <= 1e-8 * torch.linalg.norm(d)
    if restart == 100 and m.ndof <= 1000:
        assert st["lit_total"] == out[0][1]


def _with_unused(w, n):
    """The mesh with n vertices that no element uses behind its own."""
    w = dict(w)
    w["coords"] = np.concatenate([w["coords"], 100.0 + np.arange(3.0 * n).reshape(n, 3)])
    w["dir_group"] = np.concatenate([w["dir_group"], np.zeros(n, dtype=w["dir_group"].dtype)])
    return w


# rows without blocks behind the last row that has some: one, and more than the
# warps' share of one row each
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("unused", [1, 40])
def test_streamed_spmv_rows_without_blocks(fe, unused, precision):
    # the mesh without the unused vertices has the same blocks: same sums, bit for bit, and zeros
    w = W.cook(7, 5, 2, order=1, nu=0.3)
    m, mu = fe.Mesh(w), fe.Mesh(_with_unused(w, unused))
    assert mu.nnzb == m.nnzb and mu.ndof == m.ndof + 3 * unused
    rng = np.random.default_rng(11)
    d, x = (torch.from_numpy(rng.standard_normal(mu.ndof)).cuda() for _ in range(2))
    d *= 0.01
    m.tangent(d[: m.ndof].clone(), precision)
    mu.tangent(d, precision)
    y, yu = m.spmv(x[: m.ndof].clone()), mu.spmv(x, torch.full_like(x, float("nan")))
    assert torch.equal(yu[: m.ndof], y)
    assert torch.equal(yu[m.ndof:], torch.zeros_like(yu[m.ndof:]))


def _stars(n, cook):
    """n x 100 to 128 tets that share one vertex each (rows of 900 to 1,153 blocks), then Cook's membrane."""
    rng, X, T, o = np.random.default_rng(0), [], [], 0
    for i in range(n):
        k = 100 + i % 29
        x = rng.standard_normal((k, 3, 3))
        x /= np.linalg.norm(x, axis=2, keepdims=True)
        flip = np.linalg.det(x) < 0
        x[flip] = x[flip][:, [0, 2, 1]]
        X.append(np.concatenate([np.zeros((1, 3)), x.reshape(-1, 3)]))
        T.append(o + np.concatenate([np.zeros((k, 1), dtype=int), 1 + np.arange(3 * k).reshape(k, 3)], axis=1))
        o += len(X[-1])
    w = dict(W.cook(*cook, order=2, nu=0.3))
    w["tets"] = np.concatenate(T + [w["tets"] + o]).astype(w["tets"].dtype)
    w["faces"] = w["faces"] + o
    w["coords"] = np.concatenate(X + [w["coords"]])
    w["dir_group"] = np.concatenate([np.zeros(o, dtype=w["dir_group"].dtype), w["dir_group"]])
    return w


def test_streamed_spmv_empty_range(fe):
    # a row longer than a range leaves a range without rows.  Where that one
    # starts at a tile's edge and the warp has another range, the warp must
    # not walk the blocks between the two (about half of all, alone: tens of
    # milliseconds): the product takes the time of one without such rows, to
    # a factor that leaves room for anything else.
    import time
    m, p = fe.Mesh(_stars(64, (34, 34, 8))), fe.Mesh(W.cook(42, 42, 9, order=2, nu=0.3))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rp, wave = m.topology()["row_ptr"].astype(np.int64), 3 * sms * 4
    ranges = 2 * wave
    part = np.searchsorted(rp[:-1], m.nnzb * np.arange(ranges + 1) // ranges)
    empty = np.nonzero(part[:-1] == part[1:])[0]
    if not any(rp[part[e]] % 32 == 0 and e + wave < ranges for e in empty):
        pytest.skip("no such range on this device")  # (152 SMs have one)
    t = []
    for mesh in (m, p):
        x = torch.from_numpy(np.random.default_rng(12).standard_normal(mesh.ndof)).cuda()
        mesh.tangent(torch.zeros_like(x))
        y, best = mesh.spmv(x), 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            mesh.spmv(x, y)
            best = min(best, time.perf_counter() - t0)
        t.append(best)
    assert t[0] < 10 * t[1], t


# an unused vertex before, between and behind the others, clamped or not
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("group", [0, 1])
def test_tangent_with_unused_vertices(fe, group, precision):
    # the others' blocks and inverses are those of the mesh without them, bit for bit; theirs the identity
    w = W.cook(5, 4, 1, order=1, nu=0.3)
    n = len(w["coords"])
    ids = np.delete(np.arange(n + 3), [0, 17, n + 2])  # new numbers of the mesh's own vertices
    u = dict(w, tets=ids[w["tets"]].astype(w["tets"].dtype), faces=ids[w["faces"]].astype(w["faces"].dtype),
             coords=100.0 + np.arange(3.0 * (n + 3)).reshape(n + 3, 3),
             dir_group=np.full(n + 3, group, dtype=w["dir_group"].dtype))
    u["coords"][ids], u["dir_group"][ids] = w["coords"], w["dir_group"]
    m, mu = fe.Mesh(w), fe.Mesh(u)
    d = 0.01 * np.random.default_rng(13).standard_normal((n + 3, 3))
    mu.tangent(torch.from_numpy(d.reshape(-1).copy()).cuda(), precision)
    m.tangent(torch.from_numpy(d[ids].reshape(-1).copy()).cuda(), precision)
    (val, _, dinv), (valu, _, dinvu) = m.tangent_copy(), mu.tangent_copy()
    assert np.array_equal(valu, val) and np.array_equal(dinvu[ids], dinv)
    assert np.array_equal(dinvu[[0, 17, n + 2]], np.tile(np.eye(3), (3, 1, 1)))


def _device_bytes(fe, m):
    import ctypes
    info = fe.fe_mesh_info()
    assert fe.lib().fe_mesh_get_info(m.h, ctypes.byref(info)) == 0
    return info.device_bytes


def _hog(leave):
    """Tensors that leave about `leave` bytes of the device free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    out = []
    while True:
        free = torch.cuda.mem_get_info()[0] - leave
        if free < (2 << 20):
            return out
        out.append(torch.empty(min(free, 32 << 30), dtype=torch.uint8, device="cuda"))


def test_tangent_workspace_given_back(fe):
    # 128 MB of element blocks are held when the Krylov basis (117 MB) finds
    # 60 MB free: it takes their place, and the next tangents are assembled
    # without them; values and iterates as with memory to spare (FP64 tangents
    # to the parity tests' 1e-12, the iterates to the 1e-9 of the Arnoldi tests)
    w = W.cook(30, 30, 6, order=2, nu=0.3)
    m, ref = fe.Mesh(w), fe.Mesh(w)
    d = torch.from_numpy(0.01 * np.random.default_rng(14).standard_normal(m.ndof)).cuda()
    b = torch.from_numpy(np.random.default_rng(15).standard_normal(m.ndof)).cuda()
    x, y = m.zeros(), m.zeros()
    args = dict(rtol=0.0, atol=0.0, restart=100, max_it=12)
    ref.tangent(d)
    want = ref.gmres(b, **args)[0], ref.spmv(b)
    before = _device_bytes(fe, m)
    m.tangent(d)
    work = m.ne * 55 * 9 * 8
    assert _device_bytes(fe, m) - before >= work
    m.spmv(b, y)
    hog = _hog(60 << 20)
    try:
        held = _device_bytes(fe, m)
        m.gmres(b, x, **args)
        assert _device_bytes(fe, m) < held  # the basis instead of the larger workspace
        m.tangent(d)
        assert _device_bytes(fe, m) < held
        m.spmv(b, y)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.linalg.norm(x - want[0]) <= 1e-9 * torch.linalg.norm(want[0])
    assert (y - want[1]).abs().max() <= 1e-12 * want[1].abs().max()


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("case", ["cook2", "twist", "heart1"])
def test_amg_setup_without_product_lists(fe, case, precision):
    # a basis that does not fit takes the lists with it; the products are then
    # searched: the same hierarchy and V-cycle, bit for bit
    w = {"cook2": lambda: W.cook(13, 11, 5, order=2, nu=0.3), "twist": lambda: W.twist(6),
         "heart1": lambda: W.heart(nr=2, nc=24, nl=20, order=1)}[case]()
    m, ref = fe.Mesh(w), fe.Mesh(w)
    rng = np.random.default_rng(16)
    d, x = (torch.from_numpy(rng.standard_normal(m.ndof)).cuda() for _ in range(2))
    d *= 0.002
    for mesh in (m, ref):
        mesh.set_pc("amg")
        mesh.tangent(0.5 * d, precision)
    npair, npl = m.nen * (m.nen + 1) // 2, 4 if case == "twist" else 0
    work = m.ne * (9 * npair + 3 * npl * m.nen) * (8 if precision == "fp64" else 4)
    held = _device_bytes(fe, m)
    hog = _hog(20 << 20)
    try:
        with pytest.raises(fe.FEError, match="out of memory"):
            m.gmres(x, restart=1000)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert _device_bytes(fe, m) <= held - work + 4 * 8 * m.ndof - 100000  # (four vectors of the workspace fitted)
    for mesh in (m, ref):
        mesh.tangent(d, precision)
    for a, b in zip(m.amg_levels(), ref.amg_levels()):
        assert a["rho"] == b["rho"]
        assert all(np.array_equal(a[k], b[k]) for k in ("val", "pval") if k in b)
    assert torch.equal(m.pc(x), ref.pc(x))


def test_workspace_after_a_request_that_did_not_fit(fe):
    # a basis and a set of secant pairs that end in FE_ERR_OOM leave a mesh that solves as before
    w = W.cook(13, 11, 5, order=2, nu=0.3)
    m, ref = fe.Mesh(w), fe.Mesh(w)
    b = torch.from_numpy(np.random.default_rng(17).standard_normal(m.ndof)).cuda()
    opts = dict(lbfgs_m=4, ksp_restart=6, ksp_max_it=6)
    out = []
    for mesh in (m, ref):
        mesh.set_load(0.1)
        mesh.tangent(mesh.zeros())
        out.append([mesh.gmres(b, restart=6, max_it=9)[0], mesh.solve("B", mesh.zeros(), max_it=3, opts=opts)[0]])
    hog = _hog(20 << 20)
    try:
        with pytest.raises(fe.FEError, match="out of memory"):
            m.gmres(b, restart=1000)
        with pytest.raises(fe.FEError, match="out of memory"):
            m.solve("B", m.zeros(), max_it=3, opts=dict(opts, lbfgs_m=1000))
    finally:
        del hog
        torch.cuda.empty_cache()
    for mesh, o in zip((m, ref), out):
        o.append(mesh.solve("B", mesh.zeros(), max_it=3, opts=opts)[0])
        mesh.tangent(mesh.zeros())
        o.append(mesh.gmres(b, restart=6, max_it=9)[0])
    for x, y in zip(*out):
        assert torch.equal(x, y)


def test_lowsync_workspace_follows_its_own_restart(fe):
    # the low-synchronisation form's arrays belong to restarts of up to 128: a
    # longer restart of another form in between does not stand for them
    w = W.cook(9, 9, 4, order=1, nu=0.3)
    m, ref = fe.Mesh(w), fe.Mesh(w)
    b = torch.from_numpy(np.random.default_rng(18).standard_normal(m.ndof)).cuda()
    for mesh in (m, ref):
        mesh.tangent(mesh.zeros())
    for restart in (20, 300):
        m.gmres(b, restart=restart, max_it=2)
    x, y = (mesh.gmres(b, rtol=0.0, atol=0.0, restart=128, max_it=128, orthog=1)[0] for mesh in (m, ref))
    assert torch.equal(x, y)


def test_amg_levels_follow_the_last_tangent(fe):
    # an FP64 tangent, then a mixed one elsewhere on the same mesh: the levels
    # are those of the second, as on a mesh that has seen nothing else
    w = W.twist(6)
    m, ref = fe.Mesh(w), fe.Mesh(w)
    rng = np.random.default_rng(19)
    a, b = (torch.from_numpy(0.002 * rng.standard_normal(m.ndof)).cuda() for _ in range(2))
    for mesh in (m, ref):
        mesh.set_pc("amg")
    m.tangent(a, "fp64")
    first = m.amg_levels()
    m.tangent(b, "mixed_fp32")
    ref.tangent(b, "mixed_fp32")
    for f, g, r in zip(first, m.amg_levels(), ref.amg_levels()):
        for k in ("val", "pval"):
            if k in r:
                assert np.array_equal(g[k], r[k]) and not np.array_equal(g[k], f[k]), k
    m.set_pc("bj")
    m.tangent(a, "fp64")  # no hierarchy is made for this one: they stay
    for g, r in zip(m.amg_levels(), ref.amg_levels()):
        assert all(np.array_equal(g[k], r[k]) for k in ("val", "pval") if k in r)


# the waits of the forms that the limit's other test does not reach:
# compact-WY, long slices (1,644 values per block of 512 threads) and the two
# forms beyond 6,144 values per SM (956,961 unknowns on 152 SMs)
@pytest.mark.parametrize("size,orthog", [((24, 24, 20), 1), ((50, 50, 31), 2), ((68, 68, 66), 0), ((68, 68, 66), 2)])
def test_bounded_waits_of_every_form(fe, size, orthog):
    # with no polls allowed a multi-block step's waits give up, the call
    # returns FE_ERR_TIMEOUT, and the mesh then solves as before, bit for bit
    m = fe.Mesh(W.cook(*size, order=1, nu=0.3))
    m.tangent(m.zeros())
    b = torch.from_numpy(np.random.default_rng(20).standard_normal(m.ndof)).cuda()
    args = dict(rtol=0.0, atol=0.0, restart=12, max_it=12, orthog=orthog)
    x = m.gmres(b, **args)[0]
    m.set_wait_limit(0)
    with pytest.raises(fe.FEError) as e:
        m.gmres(b, **args)
    assert e.value.code == -4 and "wait" in str(e.value)
    m.set_wait_limit()
    assert torch.equal(m.gmres(b, **args)[0], x)


def _product(ptr, col, val):
    """x -> A x for block-CSR arrays."""
    n, k = len(ptr) - 1, val.shape[1]
    row = torch.from_numpy(np.repeat(np.arange(n), np.diff(ptr))).cuda()
    col, val = torch.from_numpy(col.astype(np.int64)).cuda(), torch.from_numpy(val).cuda()

    def apply(x):
        y = torch.zeros(n, k, dtype=torch.float64, device="cuda")
        return y.index_add_(0, row, torch.einsum("qij,qj->qi", val, x.view(n, k)[col])).view(-1)
    return apply


def _vcycle(levels, A0, D0, b, lv=0):
    """The V-cycle in FP64 on the hierarchy's own numbers: degree-2 Chebyshev
    steps in D^-1 A on [rho / 30, 1.1 rho] before and after the coarse
    correction, the inverse on the coarsest level."""
    L = levels[lv]
    n, k = L["n"], L["b"]
    if lv == 0:
        A, D = A0, D0
    else:
        A = _product(L["ptr"], L["col"], L["val"])
        row = np.repeat(np.arange(n), np.diff(L["ptr"]))
        D = torch.linalg.inv(torch.from_numpy(L["val"][row == L["col"]]).cuda())
    if lv == len(levels) - 1:
        return torch.linalg.solve(torch.stack([A(c) for c in torch.eye(n * k, dtype=b.dtype, device="cuda")], 1), b)
    lo, hi = L["rho"] / 30.0, 1.1 * L["rho"]
    theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
    r0 = delta / theta
    r1 = 1.0 / (2.0 / r0 - r0)

    def jac(r):
        return torch.einsum("aij,aj->ai", D, r.view(n, k)).reshape(-1)

    def smooth(x, r):
        d = jac(r) / theta
        x, r = x + d, r - A(d)
        d = r1 * r0 * d + 2.0 * r1 / delta * jac(r)
        return x + d, r - A(d)
    x, r = smooth(torch.zeros_like(b), b)
    row = torch.from_numpy(np.repeat(np.arange(n), np.diff(L["pptr"]))).cuda()
    col, pv = torch.from_numpy(L["pcol"].astype(np.int64)).cuda(), torch.from_numpy(L["pval"]).cuda()
    rc = torch.zeros(L["nc"], 6, dtype=torch.float64, device="cuda")
    rc.index_add_(0, col, torch.einsum("qij,qi->qj", pv, r.view(n, k)[row]))
    xc = _vcycle(levels, A0, D0, rc.view(-1), lv + 1).view(-1, 6)
    e = torch.zeros_like(r).view(n, k).index_add_(0, row, torch.einsum("qij,qj->qi", pv, xc[col])).view(-1)
    return smooth(x + e, r - A(e))[0]


# level 0 with several windows (more than nine tiles) and several row ranges per
# warp in both precisions, and the FP32 form of the largest meshes (16-row
# groups that fill the wave four times: from about 233,000 nodes on 152 SMs)
@pytest.mark.parametrize("size,precision,tol", [((48, 48, 8), "fp64", 1e-10), ((48, 48, 8), "mixed_fp32", 2e-3),
                                                ((64, 64, 8), "mixed_fp32", 2e-3)])
def test_vcycle_of_large_levels(fe, size, precision, tol):
    # the reference runs in FP64 on the numbers of the device's hierarchy;
    # bounds of the V-cycle's other tests
    m = fe.Mesh(W.cook(*size, order=2, nu=0.3))
    d = torch.from_numpy(0.01 * np.random.default_rng(21).standard_normal(m.ndof)).cuda()
    m.set_pc("amg")
    m.tangent(d, precision)
    b = torch.from_numpy(np.random.default_rng(22).standard_normal(m.ndof)).cuda()
    z = m.pc(b)
    top = m.topology()
    val, _, dinv = m.tangent_copy()
    want = _vcycle(m.amg_levels(), _product(top["row_ptr"], top["col"], val), torch.from_numpy(dinv).cuda(), b)
    assert (z - want).abs().max() <= tol * want.abs().max()
