"""GPU parity: every stage and the whole solve, through the C ABI, against the
CPU FP64 oracle on the same seeded inputs.

Tolerances (float64 everywhere on the FP64 path):
  * mismatch F, Jacobian entries: 1e-10 absolute (sums of a handful of O(10)
    products; only the summation order differs);
  * factorisation: ||L U - P J P^T||_max <= 1e-10 ||J||_max;
  * linear solve: ||dx - dx_oracle||_max <= 1e-8 (1 + ||dx_oracle||_max);
  * Newton result: equal status and iteration counts, |d|V|| <= 1e-6 p.u.,
    |d theta| <= 1e-6 rad, and the oracle's mismatch at the GPU's voltages
    below the tolerance 1e-8 p.u.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

torch = pytest.importorskip("torch")

from oracle import nrpf  # noqa: E402
from tests.common import case, oracle_ybus, perturbed, permuted_dense  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 1e-8


def _pf():
    import paper_2101_02270_gb300 as pf
    return pf


def _plan(g, **kw):
    return _pf().Plan.from_branches(g.n, g.f, g.t, g.r, g.x, g.b, g.bus_type, **kw)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _oracle_solve(g, S, V0, tol=TOL, maxit=10, idx=None):
    Y = oracle_ybus(g)
    idx = range(S.shape[0]) if idx is None else idx
    out = [nrpf.newton(Y, S[b], V0[b], g.bus_type, tol, maxit) for b in idx]
    return (np.array([o[0] for o in out]), np.array([o[1] for o in out]), np.array([o[2] for o in out]))


def _compare_newton(g, Vg, itg, stg, Vo, ito, sto, S, check_iters=True):
    assert np.array_equal(stg, sto)
    if check_iters:
        assert np.array_equal(itg, ito)
    ok = sto == 0
    dvm = np.abs(np.abs(Vg[ok]) - np.abs(Vo[ok]))
    dth = np.abs(np.angle(Vg[ok] * np.conj(Vo[ok])))
    assert dvm.max(initial=0) <= 1e-6 and dth.max(initial=0) <= 1e-6
    Y = oracle_ybus(g)
    _, pv, pq, _ = nrpf.bus_sets(g.bus_type)
    for b in np.flatnonzero(ok):
        F = nrpf.mismatch(Y, Vg[b], S[b], pv, pq)
        assert np.max(np.abs(F)) < TOL


@pytest.mark.parametrize("name,B", [("mesh30_b64", 64), ("mesh30_b64", 37), ("mesh2000_b10k", 45)])
def test_mismatch_stage(name, B):
    g, S, V0 = case(name, batch=B)
    V = perturbed(V0, seed=3)
    with _plan(g) as p:
        F, norm = p.stage_mismatch(_dev(S), _dev(V))
        F = F.cpu().numpy()
        norm = norm.cpu().numpy()
    Y = oracle_ybus(g)
    _, pv, pq, _ = nrpf.bus_sets(g.bus_type)
    for b in range(B):
        Fo = nrpf.mismatch(Y, V[b], S[b], pv, pq)
        assert np.max(np.abs(F[b] - Fo)) < 1e-10
        assert abs(norm[b] - np.max(np.abs(Fo))) < 1e-10


@pytest.mark.parametrize("name,B,kw", [("mesh30_b64", 40, {}), ("mesh30_b64", 33, {"ordering": "natural"}),
                                       ("mesh2000_b10k", 3, {}),
                                       ("mesh30_b64", 40, {"lu_precision": "fp32"}),
                                       ("mesh30_b64", 35, {"lu_precision": "fp32", "panel": 8}),
                                       ("mesh2000_b10k", 3, {"lu_precision": "fp32"}),
                                       ("mesh30_b64", 36, {"panel": 32}),
                                       ("mesh2000_b10k", 3, {"lu_precision": "fp32", "panel": 32}),
                                       ("mesh2000_b10k", 2, {"lu_precision": "fp32", "panel": 64}),
                                       # instance-major dense block: ndp 64 (one last panel of 64),
                                       # 320 (full, half and corner GEMM tiles), 384 (full tiles only)
                                       ("mesh30_b64", 40, {"lu_precision": "fp32", "dense_layout": "instance_major"}),
                                       ("mesh2000_b10k", 3, {"lu_precision": "fp32",
                                                             "dense_layout": "instance_major"}),
                                       ("mesh2000_b10k", 2, {"lu_precision": "fp32", "dense_layout": "instance_major",
                                                             "dense_frac": 0.12})])
def test_jacobian_and_factor_stage(name, B, kw):
    g, S, V0 = case(name, batch=B)
    V = perturbed(V0, seed=4)
    with _plan(g, **kw) as p:
        pos, colptr, rowidx = p.pattern()
        A = p.stage_factor(_dev(V), factor=False).cpu().numpy()
        LU = p.stage_factor(_dev(V), factor=True).cpu().numpy()
        m = p.info["m"]
    Y = oracle_ybus(g)
    _, pv, pq, _ = nrpf.bus_sets(g.bus_type)
    inv = np.empty(m, int)
    inv[pos] = np.arange(m)
    fp32 = kw.get("lu_precision") == "fp32"
    for b in range(B):
        J = nrpf.jacobian(Y, V[b], pv, pq).toarray()
        PJP = J[np.ix_(inv, inv)]  # row/col r of A is J row/col inv[r]
        Ag = permuted_dense(colptr, rowidx, A[b], m)
        # FP32 storage of J: relative rounding 2^-24
        assert np.max(np.abs(Ag - PJP)) < (1e-6 * np.max(np.abs(J)) if fp32 else 1e-10)
        F = permuted_dense(colptr, rowidx, LU[b], m)
        L = np.tril(F, -1) + np.eye(m)
        U = np.triu(F)
        assert np.max(np.abs(L @ U - PJP)) <= (1e-4 if fp32 else 1e-10) * np.max(np.abs(J))


@pytest.mark.parametrize("name,B,kw", [("mesh30_b64", 64, {}), ("mesh30_b64", 70, {"panel": 4}),
                                       ("mesh30_b64", 32, {"panel": 16}), ("mesh2000_b10k", 8, {}),
                                       ("mesh30_b64", 64, {"lu_precision": "fp32"}),
                                       ("mesh2000_b10k", 8, {"lu_precision": "fp32"}),
                                       ("mesh30_b64", 40, {"lu_precision": "fp32", "panel": 32}),
                                       ("mesh2000_b10k", 8, {"lu_precision": "fp32", "panel": 32}),
                                       ("mesh30_b64", 33, {"panel": 64}),
                                       ("mesh2000_b10k", 8, {"lu_precision": "fp32", "panel": 64}),
                                       ("mesh30_b64", 45, {"lu_precision": "fp32", "dense_layout": "instance_major"}),
                                       ("mesh2000_b10k", 8, {"lu_precision": "fp32",
                                                             "dense_layout": "instance_major"}),
                                       ("mesh2000_b10k", 8, {"lu_precision": "fp32", "dense_layout": "instance_major",
                                                             "dense_frac": 0.12})])
def test_linear_solve_stage(name, B, kw):
    g, S, V0 = case(name, batch=B)
    V = perturbed(V0, seed=5)
    rng = np.random.default_rng(9)
    with _plan(g, **kw) as p:
        m = p.info["m"]
        rhs = rng.standard_normal((B, m))
        dx = p.stage_linear_solve(_dev(V), _dev(rhs)).cpu().numpy()
    Y = oracle_ybus(g)
    _, pv, pq, _ = nrpf.bus_sets(g.bus_type)
    for b in range(B):
        J = nrpf.jacobian(Y, V[b], pv, pq)
        xo = spla.spsolve(J.tocsc(), rhs[b])
        tol = 1e-3 if kw.get("lu_precision") == "fp32" else 1e-8  # FP32 LU: cond(J) * 2^-24
        assert np.max(np.abs(dx[b] - xo)) <= tol * (1 + np.max(np.abs(xo)))


@pytest.mark.parametrize("B", [64, 1, 45])
def test_newton_mesh30(B):
    g, S, V0 = case("mesh30_b64", batch=B)
    with _plan(g) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    Vo, ito, sto = _oracle_solve(g, S, V0)
    _compare_newton(g, Vg, itg, stg, Vo, ito, sto, S)


def test_newton_mesh2000_ragged():
    g, S, V0 = case("mesh2000_b10k", batch=70)
    with _plan(g) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    idx = list(range(0, 70, 3))
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx])


def test_newton_mesh2000_full_batch_sampled():
    """The benchmark's launch configuration (10,000 scenarios); outputs sampled."""
    g, S, V0 = case("mesh2000_b10k")
    with _plan(g) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    idx = list(np.random.default_rng(0).choice(S.shape[0], 24, replace=False)) + [0, S.shape[0] - 1]
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx])
    # properties at any size: every instance converged, the recomputed
    # mismatch of a further sample is below tolerance
    assert np.all(stg == 0)


def test_edge_cases():
    pf = _pf()
    g, S, V0 = case("mesh30_b64", batch=8)
    Vo, ito, sto = _oracle_solve(g, S, V0, tol=1e-12, maxit=20)
    with _plan(g) as p:
        # B == 0 is a no-op
        assert pf.lib.pf_solve_batch(p._h, 0, None, None, 1e-8, 10, None, None, None, None) == 0
        # maxit = 0
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 0)
        assert np.all(it.cpu().numpy() == 0) and np.all(st.cpu().numpy() == 1)
        # starting at the solution: zero updates
        v, it, st = p.solve(_dev(S), _dev(Vo), TOL, 10)
        assert np.all(it.cpu().numpy() == 0) and np.all(st.cpu().numpy() == 0)
        # tol = 0 cannot be met: maxit updates
        v, it, st = p.solve(_dev(S), _dev(V0), 0.0, 6)
        assert np.all(it.cpu().numpy() == 6) and np.all(st.cpu().numpy() == 1)
        # a non-finite injection fails that instance only
        Sb = S.copy()
        Sb[3, 5] = np.nan
        v, it, st = p.solve(_dev(Sb), _dev(V0), TOL, 10)
        st = st.cpu().numpy()
        it = it.cpu().numpy()
        assert st[3] == 2 and it[3] == 0
        assert np.all(np.delete(st, 3) == 0)
        # bad arguments
        assert pf.lib.pf_solve_batch(p._h, -1, None, None, 1e-8, 10, None, None, None, None) == -1
        assert pf.lib.pf_solve_batch(p._h, 1, None, None, float("nan"), 10, None, None, None, None) == -1


def test_instance_major_edge_cases():
    """Instance-major FP32 dense block: a non-finite injection fails its own
    instance only, an instance that starts at the solution takes no update,
    and maxit = 0 reports every instance at its limit."""
    g, S, V0 = case("mesh2000_b10k", batch=36)
    Vo, ito, sto = _oracle_solve(g, S[:2], V0[:2], tol=1e-12, maxit=20)
    with _plan(g, lu_precision="fp32", dense_layout="instance_major") as p:
        assert p.info["dense_layout"] == 2
        Sb = S.copy()
        Sb[33, 17] = np.nan
        V0b = V0.copy()
        V0b[:2] = Vo
        v, it, st = p.solve(_dev(Sb), _dev(V0b), TOL, 20)
        st, it = st.cpu().numpy(), it.cpu().numpy()
        assert st[33] == 2 and it[33] == 0
        assert np.all(np.delete(st, 33) == 0)
        assert np.all(it[:2] == 0)
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 0)
        assert np.all(it.cpu().numpy() == 0) and np.all(st.cpu().numpy() == 1)


@pytest.mark.parametrize("n,branches,pad", [(300, 560, 128), (400, 700, 192), (800, 1300, 256), (1500, 2500, 448)])
def test_instance_major_update_far_and_near(n, branches, pad):
    """Block updates of the instance-major layout at every edge of a 128 x 128
    tile (blocks of 64 rows or columns at the end, or none) and depths of none to
    twelve chunks.  The staged solve takes the tensor cores: its steps against the
    FP64 plan's, within the factorisation's bar for FP32.  A batch whose odd
    instances start near the solution (mismatch below 1e-3, FMA updates) and
    whose even ones start flat ends at the FP64 plan's voltages."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 32)
    sc = gridgen.make_scenarios(g, 40, 0.6, 1.4)
    S, V0 = _dev(sc.sbus(g)), _dev(sc.v0_flat(g))
    with _plan(g) as p, _plan(g, lu_precision="fp32", dense_layout="instance_major") as q:
        assert q.info["dense_layout"] == 2 and q.info["dense_pad"] == pad
        F, _ = p.stage_mismatch(S, V0)
        x, y = p.stage_linear_solve(V0, F), q.stage_linear_solve(V0, F)
        assert ((y - x).norm(dim=1) / x.norm(dim=1)).max().item() < 1e-4
        V, it, st = p.solve(S, V0, TOL, 10)
        near = p.solve(S, V0, TOL, 2)[0]
        norm = p.stage_mismatch(S, near)[1]
        assert 1e-8 < norm.min().item() and norm.max().item() < 1e-3
        start = V0.clone()
        start[1::2] = near[1::2]
        v, it2, st2 = q.solve(S, start, TOL, 10)
        assert torch.all(st2 == 0) and torch.all(st == 0)
        assert torch.all(it2[1::2] <= it[1::2] - 1) and torch.all(it2[::2] == it[::2])
        assert (v - V).abs().max().item() <= 1e-6


@pytest.mark.parametrize("lu,panel", [("fp64", 4), ("fp64", 8), ("fp32", 4), ("fp32", 16)])
@pytest.mark.parametrize("B", [152 * 32, 152 * 32 + 1, 304 * 32 + 1, 456 * 32 + 1])
def test_instances_do_not_depend_on_the_batch(lu, panel, B):
    """The shapes chosen by the number of tiles (dense solves and level
    schedules) keep every instance's operations: a scenario's result in a batch
    of any size is, bit for bit, the one it has in a batch of 64."""
    g, S, V0 = case("mesh30_b64", batch=64)
    idx = np.arange(B) % 64
    with _plan(g, lu_precision=lu, panel=panel) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        v2, it2, st2 = p.solve(_dev(S[idx]), _dev(V0[idx]), TOL, 10)
    k = torch.from_numpy(idx).cuda()
    assert torch.all(st == 0)
    assert torch.equal(v2, v[k]) and torch.equal(it2, it[k]) and torch.equal(st2, st[k])


def test_singular_instance_reports_failure():
    """An instance whose Jacobian is singular (a PQ bus with zero voltage)
    stops with status 2 while the rest of the batch converges."""
    g, S, V0 = case("mesh30_b64", batch=4)
    V0 = V0.copy()
    V0[1, 7] = 0.0
    with _plan(g) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        st = st.cpu().numpy()
    assert st[1] == 2 and np.all(st[[0, 2, 3]] == 0)


def test_plan_reuse_and_capacity_growth():
    g, S, V0 = case("mesh30_b64", batch=64)
    with _plan(g, max_batch=16) as p:
        a = p.solve(_dev(S[:16]), _dev(V0[:16]), TOL, 10)
        b = p.solve(_dev(S), _dev(V0), TOL, 10)  # grows the workspace
        c = p.solve(_dev(S[:16]), _dev(V0[:16]), TOL, 10)
        assert torch.equal(a[0], c[0]) and torch.equal(a[1], c[1])
        assert torch.equal(b[0][:16], a[0])
        assert p.info["capacity"] >= 64


@pytest.mark.parametrize("name,B,panel,layout", [("mesh30_b64", 64, 0, "auto"), ("mesh2000_b10k", 40, 0, "auto"),
                                                 ("mesh2000_b10k", 40, 32, "auto"), ("mesh2000_b10k", 40, 64, "auto"),
                                                 ("mesh30_b64", 64, 0, "instance_major"),
                                                 ("mesh2000_b10k", 70, 0, "instance_major")])
def test_mixed_precision_lu(name, B, panel, layout):
    """FP32 LU + FS/BS, FP64 mismatch/update: same statuses, same tolerance,
    a few more iterations at most (default panel, the two-level panels of
    32 and 64 factorised in steps of 16, and the instance-major dense block)."""
    g, S, V0 = case(name, batch=B)
    with _plan(g, lu_precision="fp32", panel=panel, dense_layout=layout) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 20)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    idx = list(range(0, B, max(1, B // 10)))
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx], check_iters=False)
    assert np.all(itg[idx] >= ito) and np.all(itg[idx] <= ito + 3)


def test_fresh_workspace_ignores_stale_memory():
    """A plan whose workspace reuses memory freed by another plan (here full of
    NaN from a failed instance) still gives clean results: nothing of the
    solve reads workspace it did not write first."""
    g, S, V0 = case("mesh30_b64", batch=32)
    Sb = S.copy()
    Sb[:, 4] = np.nan
    with _plan(g) as p:
        p.solve(_dev(Sb), _dev(V0), TOL, 10)
        torch.cuda.synchronize()
    for _ in range(3):
        with _plan(g) as p:
            v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
            assert np.all(st.cpu().numpy() == 0)


@pytest.mark.parametrize("lu,maxit", [("fp64", 10), ("fp32", 10), ("fp64", 2)])
def test_loop_graph_matches_host_loops(lu, maxit):
    """The Newton loop run as a graph WHILE node (default), as a host loop
    ended from the host (profiled solves) and as a fixed-count loop inside a
    caller's stream capture give identical results; the graph runs one body
    per check up to the last active instance's, not maxit."""
    g, S, V0 = case("mesh30_b64", batch=64)
    Sd, Vd = _dev(S), _dev(V0)
    with _plan(g, lu_precision=lu) as p:
        outs = [tuple(torch.empty_like(t) for t in p.solve(Sd, Vd, TOL, maxit)) for _ in range(3)]
        p.profile_start([])
        p.solve(Sd, Vd, TOL, maxit, out=outs[0])
        counts = p.profile_read()
        p.profile_start(["dense_update"])
        p.solve(Sd, Vd, TOL, maxit, out=outs[1])
        p.profile_read()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            p.solve(Sd, Vd, TOL, maxit, out=outs[2])
        graph.replay()
        torch.cuda.synchronize()
    a, b, c = outs
    for x, y in ((a, b), (a, c)):
        assert torch.equal(x[0], y[0]) and torch.equal(x[1], y[1]) and torch.equal(x[2], y[2])
    st, it = a[2].cpu().numpy(), a[1].cpu().numpy()
    if maxit == 10:
        assert np.all(st == 0)
        bodies = int(it.max()) + 1  # the check that finds no instance active ends the loop
    else:
        assert np.all(st == 1) and np.all(it == maxit)
        bodies = maxit
    assert counts["check"][0] == bodies + 1  # plus the final test after the loop
    assert counts["update"][0] == bodies


@pytest.mark.parametrize("lu,B,chunk", [("fp64", 100, 32), ("fp32", 100, 0), ("fp64", 64, 64), ("fp64", 45, 200)])
def test_host_batch_chunks_match_device_solve(lu, B, chunk):
    """pf_solve_batch_host (chunks copied in and out around the solves,
    ragged last chunk) gives exactly the device-resident solve's results, and
    those match the oracle (FP64 LU: same iterations; FP32 LU: at most three
    more)."""
    g, S, V0 = case("mesh30_b64", batch=B)
    with _plan(g, lu_precision=lu) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Sh = torch.from_numpy(np.ascontiguousarray(S)).pin_memory()
        Vh = torch.from_numpy(np.ascontiguousarray(V0)).pin_memory()
        vh, ith, sth = p.solve_host(Sh, Vh, TOL, 10, chunk=chunk)
        torch.cuda.current_stream().synchronize()
        # pageable host memory works too
        vp, itp, stp = p.solve_host(torch.from_numpy(np.ascontiguousarray(S)),
                                    torch.from_numpy(np.ascontiguousarray(V0)), TOL, 10, chunk=chunk)
        torch.cuda.current_stream().synchronize()
    for a, b, c in ((v, vh, vp), (it, ith, itp), (st, sth, stp)):
        assert torch.equal(a.cpu(), b) and torch.equal(a.cpu(), c)
    # and the host-batch results against the oracle, instance by instance
    Vo, ito, sto = _oracle_solve(g, S, V0)
    ith_np = ith.numpy()
    _compare_newton(g, vh.numpy(), ith_np, sth.numpy(), Vo, ito, sto, S, check_iters=lu == "fp64")
    if lu == "fp32":
        ok = sto == 0
        assert np.all(ith_np[ok] >= ito[ok]) and np.all(ith_np[ok] <= ito[ok] + 3)


def test_host_batch_back_to_back_calls():
    """Consecutive host-batch calls without a synchronisation in between (the
    second call's copy-in overlaps the first call's solve) each return the
    device solve of their own inputs, and the oracle's solution of them."""
    g, S1, V0 = case("mesh30_b64", batch=64)
    S2 = S1 * 0.9
    with _plan(g) as p:
        ref = [p.solve(_dev(S), _dev(V0), TOL, 10) for S in (S1, S2, S1)]
        ref = [tuple(t.cpu() for t in r) for r in ref]
        hs = [torch.from_numpy(np.ascontiguousarray(S)).pin_memory() for S in (S1, S2, S1)]
        hv = torch.from_numpy(np.ascontiguousarray(V0)).pin_memory()
        outs = [p.solve_host(h, hv, TOL, 10) for h in hs]
        torch.cuda.current_stream().synchronize()
    for r, o in zip(ref, outs):
        for a, b in zip(r, o):
            assert torch.equal(a, b)
    # each call's results against the oracle on its own inputs
    for S, o in zip((S1, S2, S1), outs):
        Vo, ito, sto = _oracle_solve(g, S, V0)
        _compare_newton(g, o[0].numpy(), o[1].numpy(), o[2].numpy(), Vo, ito, sto, S)


@pytest.mark.parametrize("n,branches,lu", [(8, 10, "fp64"), (60, 85, "fp64"), (110, 140, "fp64"), (110, 140, "fp32"),
                                           (170, 215, "fp32"), (260, 330, "fp32")])
@pytest.mark.parametrize("B", [1, 33, 152 * 16 + 3])
def test_small_plan_solve(n, branches, lu, B):
    """Small plans solve each Newton step in one CTA's shared memory (32, 16 or 8
    instances of it, with and without the schedule there) and the next larger
    ones do not: voltages, iterations and status are the oracle's on sampled
    instances of every size."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=max(1, n // 10), load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, B, 0.6, 1.4)
    S, V0 = sc.sbus(g), sc.v0_flat(g)
    with _plan(g, lu_precision=lu) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    assert np.all(stg == 0)
    idx = sorted({0, B // 2, B - 1})
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx], check_iters=lu == "fp64")


@pytest.mark.parametrize("n,branches,spread", [(150, 210, 0), (190, 260, 0), (230, 330, 3), (420, 590, 0), (700, 980, 6)])
def test_fp64_update_in_fixed_point(n, branches, spread):
    """The FP64 dense block's updates of depth 16 are made in fixed point relative
    to the largest exponent of each row and column: staged solves of every size
    of the last block (8 or 16 wide) and, with impedances spread over 10^spread,
    of rows with entries far apart, are backward stable: |J x - b| at most 1e-14
    (|J| |x| + |b|), 90 units of rounding, in the max norm."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 16)
    rng = np.random.default_rng(n)
    z = 10.0 ** rng.uniform(-spread / 2, spread / 2, g.n_branch)
    g.r, g.x = g.r * z, g.x * z
    B = 36
    V = _dev(perturbed(np.broadcast_to(g.v_set.astype(complex), (B, g.n)).copy()))
    with _plan(g) as p:
        pos, colptr, rowidx = p.pattern()
        A = p.stage_factor(V, factor=False).cpu().numpy()
        m = p.info["m"]
        rhs = torch.randn(B, m, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
        x = p.stage_linear_solve(V, rhs).cpu().numpy()
    b = rhs.cpu().numpy()
    for k in range(0, B, 5):
        J = permuted_dense(colptr, rowidx, A[k], m)[np.ix_(pos, pos)]
        r = np.abs(J @ x[k] - b[k]).max()
        assert r <= 1e-14 * (np.abs(J).sum(1).max() * np.abs(x[k]).max() + np.abs(b[k]).max()), r


@pytest.mark.parametrize("n,branches,lu,kw", [(260, 330, "fp64", {}), (260, 330, "fp64", {"panel": 16}),
                                              (420, 590, "fp64", {}), (420, 590, "fp32", {}),
                                              (420, 590, "fp32", {"dense_layout": "instance_major"}),
                                              (420, 590, "fp32", {"panel": 8}), (1500, 2000, "fp64", {})])
@pytest.mark.parametrize("B", [1, 33, 64, 65])
def test_dense_block_by_clusters(n, branches, lu, kw, B):
    """Up to two tiles, the dense block is factorised and solved by a cluster of
    CTAs per instance: blocks of a few to many columns for the eight CTAs, every
    storage of the block, and the first batch beyond, against the oracle; an
    instance with a NaN injection fails alone."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, B, 0.6, 1.4)
    S, V0 = sc.sbus(g), sc.v0_flat(g)
    bad = B - 2 if B > 2 else -1
    if bad >= 0:
        S[bad, 5] = np.nan
    with _plan(g, lu_precision=lu, **kw) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
    assert np.array_equal(np.flatnonzero(stg), [bad] if bad >= 0 else []) and (bad < 0 or stg[bad] == 2)
    idx = sorted({0, B // 2, B - 1})
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx], check_iters=lu == "fp64")


@pytest.mark.parametrize("n,branches", [(30, 40), (60, 85), (150, 210), (230, 330), (420, 590), (700, 980), (900, 1300)])
@pytest.mark.parametrize("panel", [16, 32, 64])
def test_interleaved_fp32_block_by_panels(n, branches, panel):
    """The interleaved FP32 dense block, one 16-wide step up to several outer
    panels of 64, with a last panel of every number of steps and stored with more
    or less padding: staged solves are backward stable, |J x - b| at most 90 units
    of FP32 rounding times (|J| |x| + |b|) in the max norm."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=max(1, n // 10), load_scale=1 / 16)
    B = 36
    V = _dev(perturbed(np.broadcast_to(g.v_set.astype(complex), (B, g.n)).copy()))
    with _plan(g, lu_precision="fp32", panel=panel, dense_layout="interleaved") as p, _plan(g) as q:
        m = p.info["m"]
        rhs = torch.randn(B, m, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
        x = p.stage_linear_solve(V, rhs).cpu().numpy()
        pos, colptr, rowidx = q.pattern()
        A = q.stage_factor(V, factor=False).cpu().numpy()
    b = rhs.cpu().numpy()
    for k in range(0, B, 5):
        J = permuted_dense(colptr, rowidx, A[k], m)[np.ix_(pos, pos)]
        r = np.abs(J @ x[k] - b[k]).max()
        assert r <= 90 * 2.0**-24 * (np.abs(J).sum(1).max() * np.abs(x[k]).max() + np.abs(b[k]).max()), r


@pytest.mark.parametrize("n,branches", [(300, 400), (420, 590), (1000, 1500)])
def test_few_instances_of_an_interleaved_block(n, branches):
    """Up to 512 instances a solve factorises an FP32 block that is interleaved
    for its size in the instance-major form.  One workspace, batches on both sides
    of the limits, staged solves (interleaved) in between: every solve has the
    oracle's voltages, a NaN injection fails alone, and a batch solved again after
    the others has the same result, bit for bit."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, 513, 0.6, 1.4)
    S, V0 = sc.sbus(g), sc.v0_flat(g)
    S[40, 5] = np.nan
    idx = [0, 39, 41, 64]
    Vo, ito, sto = _oracle_solve(g, S, V0, idx=idx)
    first = {}
    with _plan(g, lu_precision="fp32") as p:
        assert p.info["dense_layout"] == 1
        for B in (513, 65, 512, 513, 65):
            v, it, st = p.solve(_dev(S[:B]), _dev(V0[:B]), TOL, 10)
            Vg, itg, stg = v.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()
            assert np.array_equal(np.flatnonzero(stg), [40]) and stg[40] == 2
            _compare_newton(g, Vg[idx], itg[idx], stg[idx], Vo, ito, sto, S[idx], check_iters=False)
            f = first.setdefault(B, (Vg, itg))
            assert np.array_equal(f[0], Vg, equal_nan=True) and np.array_equal(f[1], itg)
            x = p.stage_linear_solve(v[:36], torch.ones(36, p.info["m"], dtype=torch.float64, device="cuda"))
            assert torch.isfinite(x).all()


def test_launch_counts_of_batches_on_different_kernels():
    """Which kernels an iteration launches depends on the batch (a cluster per
    instance up to two tiles, sparse columns instead of entries beyond 152, per
    loop graph): the counts of one plan that solves several sizes are the sum
    of the counts of plans that solve one each."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=300, n_branch=400, n_pv=30, load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, 152 * 32 + 1, 0.6, 1.4)
    S, V0 = _dev(sc.sbus(g)), _dev(sc.v0_flat(g))
    total = {}
    for B in (64, len(S)):
        with _plan(g) as p:
            p.profile_start([])
            p.solve(S[:B], V0[:B], TOL, 10)
            one = {k: c[0] for k, c in p.profile_read().items()}
        for k, c in one.items():
            total[k] = total.get(k, 0) + (2 * c if B == 64 else c)
    assert total["dense_update"] > 0 and total["lu_sparse_level"] > 0
    with _plan(g) as p:
        p.solve(S, V0, TOL, 10)  # the workspace of the largest batch, so that no graph is made anew
        p.profile_start([])
        for B in (64, len(S), 64):
            p.solve(S[:B], V0[:B], TOL, 10)
        assert {k: c[0] for k, c in p.profile_read().items()} == total


def test_more_batch_sizes_than_loop_graphs():
    """A plan keeps 64 loop graphs; further batch sizes start the set over, with
    the same results and every launch counted."""
    g, S, V0 = case("mesh30_b64", batch=64)
    idx = np.arange(70 * 32) % 64
    with _plan(g) as p:
        v, it, st = p.solve(_dev(S), _dev(V0), TOL, 10)
        Sd, Vd, k = _dev(S[idx]), _dev(V0[idx]), torch.from_numpy(idx).cuda()
        p.solve(Sd, Vd, TOL, 10)
        p.profile_start([])
        for t in range(1, 71):
            w, it2, st2 = p.solve(Sd[:32 * t], Vd[:32 * t], TOL, 10)
            assert torch.equal(w, v[k[:32 * t]]) and torch.equal(it2, it[k[:32 * t]])
        counts = p.profile_read()
    assert counts["update"][0] == 70 * (int(it.max()) + 1)


@pytest.mark.parametrize("n,branches,lu,waves", [(55, 75, "fp64", 16), (85, 116, "fp64", 8), (40, 50, "fp32", 32),
                                                 (55, 69, "fp32", 0), (120, 164, "fp32", 0), (30, 41, "fp64", None),
                                                 (30, 41, "fp32", None), (50, 63, "fp64", 32)])
def test_small_plans_leave_their_kernel_beyond_one_wave(n, branches, lu, waves):
    """A batch of more than `waves` instances per SM (as many as fit a CTA, or two CTAs'
    where a plan has few values and many levels) goes from the small plans' kernel to
    the level kernels, larger FP32 plans always, the smallest plans never.  Voltages on
    either side of the line are those of the same scenarios within a few units of
    rounding."""
    import gridgen
    g = gridgen.make_grid("mesh30_b64" if n < 100 else "mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10,
                          load_scale=1 / 16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    last = 32 * (sms * (waves or 0) // 32) or 64
    sc = gridgen.make_scenarios(g, last + 1 if waves else 33 * sms, 0.6, 1.4)
    S, V0 = _dev(sc.sbus(g)), _dev(sc.v0_flat(g))
    with _plan(g, lu_precision=lu) as p:
        out = []
        for B in (last, len(S)):
            p.profile_start([])
            out.append(p.solve(S[:B], V0[:B], TOL, 10))
            levels = p.profile_read()["bwd_level"][0] > 0
            assert levels == (waves is not None and B > sms * waves)
    a, b = out
    assert torch.all(a[2] == 0) and torch.all(b[2] == 0) and torch.equal(a[1], b[1][:last])
    assert (a[0] - b[0][:last]).abs().max().item() < (1e-12 if lu == "fp64" else 1e-9)


@pytest.mark.parametrize("n,branches,lu,inside,beyond", [(2000, 2900, "fp32", 8, 32), (2000, 2900, "fp64", 8, 64),
                                                         (2000, 2600, "fp32", 32, 33), (600, 888, "fp32", 64, 65),
                                                         (1000, 1300, "fp64", 64, 65)])
def test_clusters_where_they_are_resident(n, branches, lu, inside, beyond):
    """The dense block goes to a cluster per instance while the batch's clusters fit
    the GPU (about; FP64 twice over), however many tiles that is: wide blocks
    only for a few instances.  Instances have the same voltages on both sides."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 32)
    sc = gridgen.make_scenarios(g, beyond, 0.6, 1.4)
    S, V0 = _dev(sc.sbus(g)), _dev(sc.v0_flat(g))
    out = {}
    with _plan(g, lu_precision=lu) as p:
        for B in (inside, beyond):
            p.profile_start([])
            out[B] = p.solve(S[:B], V0[:B], TOL, 10)
            assert (p.profile_read()["dense_update"][0] == 0) == (B == inside)
    a, b = out[inside], out[beyond]
    assert torch.all(a[2] == 0) and torch.all(b[2] == 0)
    assert (a[0] - b[0][:inside]).abs().max().item() < (1e-12 if lu == "fp64" else 1e-9)


@pytest.mark.parametrize("lu,B,chunk", [("fp64", 200, 32), ("fp64", 65, 64), ("fp32", 600, 512), ("fp32", 600, 64),
                                        ("fp32", 300, 40), ("fp64", 64, 32)])
def test_host_chunks_take_the_kernels_of_the_batch(lu, B, chunk):
    """On a grid whose batches of up to 64 and up to 512 instances take kernels of
    their own: a batch from host memory in chunks of such sizes still gives the
    device-resident solve's results, bit for bit."""
    import gridgen
    g = gridgen.make_grid("mesh2000_b10k", 0, n=420, n_branch=590, n_pv=42, load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, B, 0.6, 1.4)
    S, V0 = (torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in (sc.sbus(g), sc.v0_flat(g)))
    with _plan(g, lu_precision=lu) as p:
        h = p.solve_host(S, V0, TOL, 10, chunk=chunk)
        torch.cuda.synchronize()
        d = p.solve(S.cuda(), V0.cuda(), TOL, 10)
    assert torch.all(d[2] == 0)
    for x, y in zip(h, d):
        assert torch.equal(x, y.cpu())
