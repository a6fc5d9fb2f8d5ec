"""The forms that a launch picks by size, on both sides of the lines between
them: the node-by-node operator up to 64^3 and the march above (ragged tiles),
the right-hand side with its boundary rows in one launch up to 64^3 and in two
above, transfers on grids that end inside a tile."""
import numpy as np
import pytest

import oracle
from paper_1901_05118_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1901_05118_gb300 import binding as B  # noqa: E402

DEV = torch.device("cuda", 0)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def rel_max(got, ref):
    return float(np.abs(got - ref).max() / np.abs(ref).max())


@pytest.mark.parametrize("n,bc_kind", [(6, 1), (64, 2), (65, 1), (66, 2), (98, 1), (129, 2)])
def test_operator_overwrites_every_entry(n, bc_kind):
    u = P.random_field(n, 400 + n)
    y = torch.full((n + 1,) * 3, float("nan"), dtype=torch.float64, device=DEV)
    B.stencil_apply(B.Level(n, bc_kind), dev(u), y)
    assert rel_max(y.cpu().numpy(), oracle.stencil_apply(n, bc_kind, u)) <= 1e-12


@pytest.mark.parametrize("n,stride", [(5, 1), (9, 2), (64, 1), (65, 1), (70, 2)])
@pytest.mark.parametrize("bc_kind", [1, 2])
def test_right_hand_side(n, stride, bc_kind):
    ns = n * stride
    f, g1 = P.random_field(ns, 410), P.random_field(ns, 411)
    g2 = np.random.Generator(np.random.PCG64(412)).uniform(-1, 1, size=(6, ns + 1, ns + 1))
    fh = B.excmg_assemble_rhs(B.Level(n, bc_kind), ns, dev(f), dev(g1), dev(g2)).cpu().numpy()
    ref = oracle.assemble_rhs(n, bc_kind, oracle.inject_nodes(ns, stride, f), oracle.inject_nodes(ns, stride, g1),
                              oracle.inject_faces(ns, stride, g2))
    assert np.abs(fh - ref).max() <= 1e-13 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("nf", [12, 28, 64, 68, 100])
def test_transfers(nf):
    u1, u0, uh = P.random_field(nf // 2, 420), P.random_field(nf // 4, 421), P.random_field(nf, 422)
    w = B.extrapolate_interpolate(nf, dev(u1), dev(u0)).cpu().numpy()
    assert rel_max(w, oracle.exp_finite(nf, u1, u0)) <= 1e-13
    ut = B.midpoint_extrapolate(nf, dev(uh), dev(u1)).cpu().numpy()
    assert rel_max(ut, oracle.exp_true(nf, uh, u1)) <= 1e-13


def test_start_from_a_guess_in_the_separate_schedule():
    """The march that stores b - A u alone (the other schedule forms its
    copies with it): three iterations from a nonzero guess, within the bound that
    the repository's fixed-iteration comparisons have."""
    n = 98
    b, x0 = P.random_field(n, 81), P.random_field(n, 82)
    ctx = B.Context(DEV)
    ctx.set_schedule("separate")
    x = dev(x0)
    it, rel, rc = B.bicg_solve(B.Level(n, 1, ctx), dev(b), x, 0.0, 3)
    xr, itr, relr, rcr = oracle.bicg(n, 1, b, x0, 0.0, max_iter=3)
    assert it == itr == 3
    assert rel_max(x.cpu().numpy(), xr) <= 1e-10


@pytest.mark.parametrize("n,dim", [(122, 3), (123, 3), (1365, 2), (1366, 2)])
@pytest.mark.parametrize("mode", ["full", "elided"])
def test_vector_kernels_on_both_sides_of_their_line(n, dim, mode):
    """Twelve grid strides (1867776 entries) lie between each pair of sizes:
    one entry per thread at a time below, two from there on."""
    entries = (n + 1) ** dim
    assert (entries >= 12 * 152 * 4 * 256) == (n in (123, 1366))
    ctx = B.Context(DEV)
    ctx.set_shadow_mode(mode)
    ctx.set_schedule("separate")
    if dim == 3:
        b, x0 = P.random_field(n, 85), P.random_field(n, 86)
        x = dev(x0)
        B.bicg_solve(B.Level(n, 2, ctx), dev(b), x, 0.0, 3)
        xr = oracle.bicg(n, 2, b, x0, 0.0, max_iter=3)[0]
    else:
        b, x0 = P.random_field_2d(n, 85), P.random_field_2d(n, 86)
        x = dev(x0)
        B.bicg_solve2d(n, 2, dev(b), x, 0.0, 3, ctx=ctx)
        xr = oracle.bicg2d(n, 2, b, x0, 0.0, max_iter=3)[0]
    assert rel_max(x.cpu().numpy(), xr) <= 1e-10


@pytest.mark.parametrize("n", [72, 90])
@pytest.mark.parametrize("schedule", ["separate", "fused"])
def test_given_shadow_that_is_the_residual(n, schedule):
    """r*_0 = r_0 given by the caller, with anything on its boundary nodes: A p serves
    A^T p* as in a call without r*_0 (the bytes per launch say so), an r*_0 that differs at one
    node has its own.  Iterates as in the repository's fixed-iteration comparisons."""
    b = P.random_field(n, 87)
    ctx = B.Context(DEV)
    ctx.set_schedule(schedule)
    ctx.profile()
    lvl = B.Level(n, 1, ctx)
    moved = {}
    for what in ("same", "one node off"):
        shadow = b.copy()
        if what != "same":
            shadow[n // 2, n // 3, 1] *= 1 + 2.0 ** -40
        ctx.profile()   # clears the records
        x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
        it, _, _ = B.bicg_solve(lvl, dev(b), x, 0.0, 4, shadow=dev(shadow))
        _, launches, moved[what] = ctx.profile_read(n)
        assert it == launches == 4
        xr = oracle.bicg(n, 1, b, np.zeros_like(b), 0.0, max_iter=4)[0]
        assert rel_max(x.cpu().numpy(), xr) <= 1e-10
    fields = 4 * 3 if schedule == "separate" else 3 + 3 * 7
    assert moved["same"] == fields * 8.0 * (n - 1) ** 3
    assert moved["one node off"] == moved["same"] + 4 * 8.0 * (n - 1) ** 3


@pytest.mark.parametrize("n", [65, 81, 82])
@pytest.mark.parametrize("schedule", ["separate", "fused"])
def test_operator_timing_has_launches_above_64(n, schedule):
    """Every iteration's operator launch is timed from 65^3 on, also where the
    call runs on chip without timing; the iterates are those of either path within
    the bound of the repository's fixed-iteration comparisons."""
    b = dev(P.random_field(n, 88))
    got = []
    for timed in (False, True):
        ctx = B.Context(DEV)
        ctx.set_schedule(schedule)
        ctx.profile(timed)
        x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
        it, _, _ = B.bicg_solve(B.Level(n, 1, ctx), b, x, 0.0, 7)
        assert it == 7
        ms, launches, moved = ctx.profile_read(n)
        assert launches == (7 if timed else 0)
        if timed:
            fields = 7 * 3 if schedule == "separate" else 3 + 6 * 7
            assert ms > 0 and moved == fields * 8.0 * (n - 1) ** 3
        got.append(x.cpu().numpy())
    assert rel_max(got[1], got[0]) <= 1e-10
