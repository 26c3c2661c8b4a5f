"""A GPU with no memory to spare: scratch that only makes solves faster is left out,
and what fits without it is solved, with per-instance admittances and from host memory
too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gridgen  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lu", ["fp64", "fp32"])
def test_optional_scratch_leaves_what_the_plan_needs_later(lu):
    import paper_2101_02270_gb300 as pf

    n, B = 420, 6000
    g = gridgen.make_grid("mesh2000_b10k", 0, n=n, n_branch=590, n_pv=42, load_scale=1 / 16)
    sc = gridgen.make_scenarios(g, B, 0.6, 1.4)
    S, V0 = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.sbus(g), sc.v0_flat(g)))
    out = (torch.empty_like(S), torch.empty(B, dtype=torch.int32, device="cuda"),
           torch.empty(B, dtype=torch.uint8, device="cuda"))
    Sh, Vh = S.cpu().pin_memory(), V0.cpu().pin_memory()
    host = (torch.empty_like(Sh).pin_memory(), torch.empty(B, dtype=torch.int32).pin_memory(),
            torch.empty(B, dtype=torch.uint8).pin_memory())

    def plan():
        return pf.Plan.from_branches(g.n, g.f, g.t, g.r, g.x, g.b, g.bus_type, lu_precision=lu)

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    with plan() as p:
        info = p.info
        Y = torch.from_numpy(np.repeat(p.ybus_values(), B, 0)).cuda()
        before = free()
        p.solve(S, V0, 1e-8, 10, out=out)
        taken = before - free()
        ref = out[0].cpu()
        assert torch.all(out[2] == 0)
        few = p.solve(S[:300], V0[:300], 1e-8, 10)[0].cpu()
    with plan() as p:
        Bp = (B + 31) // 32 * 32
        width, ndp = (8, info["dense_pad"]) if lu == "fp64" else (4, 0)
        if lu == "fp64":  # operands in fixed point, inverse pivots of 152 tiles
            optional = Bp // 32 * (info["dense_pad"] // 4 * 64 * 33 * 16) + info["sparse_cols"] * 8 * 152 * 32
        else:  # inverse pivots, inverses for 512 instances
            optional = info["sparse_cols"] * 4 * Bp + 512 * 32768
        later = Bp * 16 * info["nnz_ybus"] + 2 * B * (48 * n + 5)
        assert optional > 24 << 20
        need = taken - optional + later + (12 << 20)  # a few MB for the allocations' granularity
        held = torch.empty(free() - need, dtype=torch.uint8, device="cuda")
        tol = 1e-12 if lu == "fp64" else 1e-9

        def check(v, status, expected):
            assert torch.all(status.cpu() == 0) and (v.cpu() - expected).abs().max().item() < tol

        try:
            p.solve(S, V0, 1e-8, 10, out=out)
            check(out[0], out[2], ref)
            p.solve_y(Y, S, V0, 1e-8, 10, out=out)
            check(out[0], out[2], ref)
            p.solve_host(Sh, Vh, 1e-8, 10, out=host)
            torch.cuda.synchronize()
            check(host[0], host[2], ref)
            # few instances without the scratch of their kernels
            p.solve(S[:300], V0[:300], 1e-8, 10, out=tuple(o[:300] for o in out))
            check(out[0][:300], out[2][:300], few)
        finally:
            del held
            torch.cuda.empty_cache()
