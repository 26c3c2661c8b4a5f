"""The FP64 trailing update in fixed point on badly scaled grids: row by row, against
the same solves with multiply-adds (panel 16 has no fixed-point form)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gridgen  # noqa: E402
from tests.common import permuted_dense, perturbed  # noqa: E402

pytestmark = pytest.mark.gpu


def _plan(g, **kw):
    import paper_2101_02270_gb300 as pf
    return pf.Plan.from_branches(g.n, g.f, g.t, g.r, g.x, g.b, g.bus_type, **kw)


def _grid(n, branches, kind, spread):
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=branches, n_pv=n // 10, load_scale=1 / 16)
    rng = np.random.default_rng(n + spread)
    z = 10.0 ** rng.uniform(-spread / 2, spread / 2, g.n_branch) if kind == "wide" else \
        np.where(rng.random(g.n_branch) < 0.03, 10.0 ** -spread, 1.0)
    g.r, g.x = g.r * z, g.x * z
    return g


@pytest.mark.parametrize("n,branches", [(230, 330), (420, 590), (700, 980)])
@pytest.mark.parametrize("kind,spread", [("wide", 0), ("wide", 6), ("wide", 8), ("short", 2), ("short", 4), ("short", 8)])
def test_rows_are_as_accurate_as_by_multiply_adds(n, branches, kind, spread):
    """Component-wise backward error max_i |J x - b|_i / (|J| |x| + |b|)_i of staged
    solves, impedances spread over 10^spread or 3 % of the lines shorter by it.  Both
    forms round about as often, at other places.  Of one instance that alone can
    change the error several times (multiply-adds in reversed order: up to 5 in 33
    draws), so the mean over 33 instances is compared, to a factor of 2, and the worst
    of one form with the worst of the other, to 8."""
    g = _grid(n, branches, kind, spread)
    B = 33
    V = torch.from_numpy(perturbed(np.broadcast_to(g.v_set.astype(complex), (B, g.n)).copy())).cuda()
    err = {}
    for panel in (8, 16):
        with _plan(g, panel=panel) as p:
            m = p.info["m"]
            pos, colptr, rowidx = p.pattern()
            A = p.stage_factor(V, factor=False).cpu().numpy()
            rhs = torch.randn(B, m, dtype=torch.float64, device="cuda",
                              generator=torch.Generator("cuda").manual_seed(n))
            x = p.stage_linear_solve(V, rhs).cpu().numpy()
        b = rhs.cpu().numpy()
        e = np.empty(B)
        for k in range(B):
            J = permuted_dense(colptr, rowidx, A[k], m)[np.ix_(pos, pos)]
            r = np.abs((J.astype(np.longdouble) @ x[k].astype(np.longdouble) - b[k]).astype(float))
            e[k] = (r / (np.abs(J) @ np.abs(x[k]) + np.abs(b[k]))).max()
        err[panel] = e
    ratio = err[8] / err[16]
    assert np.exp(np.log(ratio).mean()) < 2 and err[8].max() < 8 * err[16].max()


def test_an_instance_does_not_depend_on_its_tile():
    """Half of the instances have lines shorter by 10^4, which they are too widely
    scaled for fixed point with: the others' results are, bit for bit, those that
    they have among their like."""
    n, branches = 300, 420
    g, h = _grid(n, branches, "wide", 0), _grid(n, branches, "short", 4)
    sc = gridgen.make_scenarios(g, 96, 0.9, 1.1)
    S, V0 = (torch.from_numpy(a).cuda() for a in (sc.sbus(g), sc.v0_flat(g)))
    with _plan(g) as p, _plan(h) as q:
        yg, yh = (torch.from_numpy(np.broadcast_to(t.ybus_values(np.ones((1, branches), bool)), (96, p.info["nnz_ybus"]))
                                   .copy()).cuda() for t in (p, q))
        a = p.solve_y(yg, S, V0, 1e-8, 10)
        yg[1::2] = yh[1::2]
        b = p.solve_y(yg, S, V0, 1e-8, 10)
        c = q.solve(S, V0, 1e-8, 10)
    assert torch.all(a[2] == 0) and torch.all(b[2] == 0)
    assert torch.equal(a[0][::2], b[0][::2]) and torch.equal(a[1][::2], b[1][::2])
    # the others: solutions of the grid with the short lines, whose plan has another order
    assert (b[0][1::2] - c[0][1::2]).abs().max().item() < 1e-7
