"""The kernels that a batch's size selects: every one's linear solve by itself, and no
dependence on the size within one of them."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

torch = pytest.importorskip("torch")

import gridgen  # noqa: E402
from oracle import nrpf  # noqa: E402
from tests.common import oracle_ybus  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 1e-8


def _plan(g, **kw):
    import paper_2101_02270_gb300 as pf
    return pf.Plan.from_branches(g.n, g.f, g.t, g.r, g.x, g.b, g.bus_type, **kw)


def _case(n, branches, B):
    g = gridgen.make_grid("mesh30_b64" if n < 100 else "mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=max(1, n // 10),
                          load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, B, 0.6, 1.4)
    return g, sc.sbus(g), sc.v0_flat(g)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (buses, branches, LU, options, instances): classes launched, classes not launched
ROUTES = [
    ((30, 41, "fp64", {}, 64), [], ["fwd_level", "dense_solve"]),                      # one CTA's shared memory
    ((40, 50, "fp32", {}, 64), [], ["fwd_level", "dense_solve"]),
    ((420, 590, "fp64", {}, 1), ["fwd_level", "dense_solve"], ["dense_update"]),       # a cluster per instance
    ((420, 590, "fp64", {}, 64), ["fwd_level", "dense_solve"], ["dense_update"]),
    ((420, 590, "fp32", {}, 33), ["fwd_level", "dense_solve"], ["dense_update"]),
    ((420, 590, "fp32", {"dense_layout": "instance_major"}, 33), ["dense_solve"], ["dense_update"]),
    ((420, 590, "fp32", {}, 65), ["dense_panel"], []),                                 # instance-major, for few instances
    ((700, 980, "fp32", {}, 512), ["dense_update"], []),
    ((700, 980, "fp32", {}, 513), ["dense_update"], []),                               # interleaved
    ((700, 980, "fp32", {"dense_layout": "instance_major"}, 70), ["dense_update"], []),
    ((420, 590, "fp64", {}, 65), ["dense_update"], []),                                # fixed point
    ((420, 590, "fp64", {"panel": 16}, 65), ["dense_update"], []),                     # multiply-adds
]


@pytest.mark.parametrize("case,launched,absent", ROUTES)
def test_first_newton_step_of_every_route(case, launched, absent):
    """One Newton update from a flat start: the step that the batch's kernels make is
    the sparse direct solver's, to 1e-10 of its norm in FP64 (rounding times a condition
    number of 10^4 to 10^5) and to 1e-4 in FP32."""
    n, branches, lu, kw, B = case
    g, S, V0 = _case(n, branches, B)
    with _plan(g, lu_precision=lu, **kw) as p:
        p.profile_start([])
        V, it, st = p.solve(_dev(S), _dev(V0), TOL, 1)
        counts = p.profile_read()
    assert all(counts[c][0] > 0 for c in launched) and all(counts[c][0] == 0 for c in absent)
    assert torch.all(it == 1)
    V = V.cpu().numpy()
    Y = oracle_ybus(g)
    _, pv, pq, _ = nrpf.bus_sets(g.bus_type)
    pvpq = np.concatenate([pv, pq])
    for b in sorted({0, B // 2, B - 1}):
        F = nrpf.mismatch(Y, V0[b], S[b], pv, pq)
        dx = -spla.spsolve(nrpf.jacobian(Y, V0[b], pv, pq).tocsc(), F)
        got = np.concatenate([np.angle(V[b] * np.conj(V0[b]))[pvpq], (np.abs(V[b]) - np.abs(V0[b]))[pq]])
        assert np.linalg.norm(got - dx) <= (1e-10 if lu == "fp64" else 1e-4) * np.linalg.norm(dx), b


@pytest.mark.parametrize("n,branches,lu,kw", [(300, 400, "fp64", {}), (300, 400, "fp64", {"panel": 16}),
                                              (300, 400, "fp32", {}), (300, 400, "fp32", {"panel": 8})])
def test_level_kernels_do_not_depend_on_the_batch(n, branches, lu, kw):
    """Beyond the few-instance kernels the shapes of the level schedules and of the
    dense solve, and in FP64 entries or columns for the sparse part, change at 152,
    304 and 456 tiles: a scenario's result is the same, bit for bit, on every side."""
    g, S, V0 = _case(n, branches, 600)
    top = 456 * 32 + 1
    idx = np.arange(top) % 600
    Sd, Vd = _dev(S[idx]), _dev(V0[idx])
    k = torch.from_numpy(idx).cuda()
    with _plan(g, lu_precision=lu, **kw) as p:
        v, it, st = p.solve(Sd[:600], Vd[:600], TOL, 10)
        assert torch.all(st == 0)
        for B in (152 * 32, 152 * 32 + 1, 304 * 32, 304 * 32 + 1, 456 * 32, top):
            p.profile_start([])
            v2, it2, st2 = p.solve(Sd[:B], Vd[:B], TOL, 10)
            counts = p.profile_read()
            bodies = counts["update"][0]
            assert counts["fwd_level"][0] == counts["bwd_level"][0] == bodies > 0
            by_columns = lu == "fp64" and B > 152 * 32
            assert (counts["lu_sparse_level"][0] > bodies) == by_columns
            assert torch.equal(v2, v[k[:B]]) and torch.equal(it2, it[k[:B]]) and torch.equal(st2, st[k[:B]])
