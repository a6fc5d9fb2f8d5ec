"""The resident Bi-CG kernels (grids up to 81^3, every vector on chip) at the
edges of their brick decompositions: smallest and largest grids, bricks cut
short by the boundary, one to eight nodes per thread, a call longer than one
launch, the FP32 correction solves."""
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


@pytest.mark.parametrize("n,bc_kind,iters", [(4, 1, 9), (5, 2, 12), (9, 1, 20), (14, 2, 20), (23, 1, 20), (33, 2, 20),
                                             (41, 1, 20), (47, 2, 20), (53, 1, 20), (58, 2, 20), (63, 1, 20), (65, 2, 20),
                                             (64, 2, 20), (67, 1, 20), (74, 2, 20), (81, 1, 20), (82, 2, 20)])
def test_iterates_match_the_oracle(n, bc_kind, iters):
    """Fixed iteration counts from random data: entry by entry within the
    1e-10 that a few dozen FP64 Bi-CG steps in another summation order keep."""
    b = P.random_field(n, 301)
    x0 = P.random_field(n, 302) * 0.1
    x = dev(x0)
    it, rel, _ = B.bicg_solve(B.Level(n, bc_kind), dev(b), x, 0.0, iters)
    xr, itr, relr, _ = oracle.bicg(n, bc_kind, b, x0, 0.0, max_iter=iters)
    assert it == itr == iters
    assert rel == pytest.approx(relr, rel=1e-8)
    assert rel_max(x.cpu().numpy(), xr) <= 1e-10


@pytest.mark.parametrize("n,bc_kind,iters", [(4, 2, 5), (9, 1, 20), (31, 2, 20), (97, 1, 20), (200, 2, 20),
                                             (333, 1, 20), (512, 2, 20), (513, 1, 20)])
def test_2d_iterates_match_the_oracle(n, bc_kind, iters):
    """The 2D form, up to its largest grid and one beyond it."""
    b = P.random_field_2d(n, 305)
    x0 = P.random_field_2d(n, 306) * 0.1
    x = dev(x0)
    it, rel, _ = B.bicg_solve2d(n, bc_kind, dev(b), x, 0.0, iters)
    xr, itr, relr, _ = oracle.bicg2d(n, bc_kind, b, x0, 0.0, max_iter=iters)
    assert it == itr == iters
    assert rel == pytest.approx(relr, rel=1e-8)
    assert rel_max(x.cpu().numpy(), xr) <= 1e-10


def test_call_longer_than_one_launch():
    """1100 iterations of one call (a launch takes up to 1024): the residual
    of the recurrence, carried over from launch to launch, is still the true
    residual.  The two part by rounding of the order eps |A| |x| / |b| <
    eps cond = 3e-11 here, times a growth factor; had a vector or scalar not
    been carried over, they would part by the residual itself."""
    n = 30
    b = P.random_field(n, 303)
    b[[0, -1]] = 0
    b[:, [0, -1]] = 0
    b[:, :, [0, -1]] = 0
    lvl = B.Level(n, 1)
    tb = dev(b)
    x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
    it, rel, rc = B.bicg_solve(lvl, tb, x, 0.0, 1100)
    assert it == 1100 and rc == -4
    true = float((tb - B.stencil_apply(lvl, x)).norm() / tb.norm())
    assert abs(true - rel) <= 1e-8


def test_general_kernel_where_the_budget_has_no_room():
    """A budget that holds the Bi-CG vectors but not the exchange words: the
    call still runs, on the general cooperative kernel."""
    n = 40
    b = P.random_field(n, 304)
    want = None
    for budget in (0, 6 * 8 * (n + 1) ** 3):
        x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
        ctx = B.Context(hbm_budget_bytes=budget)
        B.bicg_solve(B.Level(n, 2, ctx), dev(b), x, 0.0, 20)
        if budget:
            assert ctx.bytes <= budget
        got = x.cpu().numpy()
        want = got if want is None else want
        assert rel_max(got, want) <= 1e-10


@pytest.mark.parametrize("n,nc,bc_kind", [(16, 4, 1), (28, 7, 2), (40, 5, 1), (64, 8, 2)])
def test_mixed_levels(n, nc, bc_kind):
    """FP32 correction solves on resident levels: what the mixed solve promises
    is an FP64 residual below the tolerance on every level; on the finest one
    it is formed again here from u_h."""
    prob = P.exp_sum()
    f, g1, g2 = (dev(a) for a in prob.data(n, bc_kind))
    uh = torch.empty((n + 1,) * 3, dtype=torch.float64, device=DEV)
    _, stats = B.excmg_solve(n, nc, bc_kind, f, g1, g2, 1e-10, u_h_out=uh, return_stats=True, precision="mixed")
    for s in stats[2:]:
        assert s["relres"] <= 1e-10 and not s["stagnated"]
    lvl = B.Level(n, bc_kind)
    fh = B.excmg_assemble_rhs(lvl, n, f, g1, g2)
    rel = float((fh - B.stencil_apply(lvl, uh)).norm() / fh.norm())
    assert rel <= 1e-10 * (1 + 1e-3)


def test_batch_large_level_is_not_kept_out():
    """A 64^3 level needs most of the SMs at once; a stream of 32^3 requests
    that takes every SM as it comes free must not keep it waiting.  Each of
    its Bi-CG calls may wait 20 ms plus one launch of a small level, in which
    the stream finishes some 100 requests: 2000 are a wide margin."""
    prob = P.by_name("random_sines:4")
    big, small = ([dev(a) for a in prob.data(n, 2)] for n in (64, 32))
    batch = B.Batch(max_instances=16)
    ident, _ = batch.submit(64, 8, 2, *big, 1e-8, precision="fp64")
    live = [batch.submit(32, 4, 2, *small, 1e-10, precision="fp64")[0] for _ in range(13)]
    done = 0
    while not batch.query(ident)["done"] and done < 2000:
        batch.step()
        left = [k for k in live if not batch.query(k)["done"]]
        done += len(live) - len(left)
        live = left + [batch.submit(32, 4, 2, *small, 1e-10, precision="fp64")[0] for _ in range(13 - len(left))]
    assert batch.query(ident)["done"]
    batch.run()


def _operator_ld(n, bc_kind, v):
    """A_h on interior values v[k, j, i] in numpy's extended precision."""
    m = n - 1
    pad = np.zeros((m + 4,) * 3, dtype=np.longdouble)
    pad[2:-2, 2:-2, 2:-2] = v

    def at(*o):
        return pad[tuple(slice(2 + a, 2 + a + m) for a in o)]

    end = np.zeros(m, dtype=np.longdouble)
    end[0] += 1
    end[-1] += 1
    faces = end[:, None, None] + end[None, :, None] + end[None, None, :]
    y = (42 + (1 if bc_kind == 1 else -1) * faces) * at(0, 0, 0)
    for a in range(3):
        for s in (-1, 1):
            o = [0, 0, 0]
            o[a] = s
            y = y - 12 * at(*o)
            o[a] = 2 * s
            y = y + at(*o)
        for b in range(a + 1, 3):
            for s in (-1, 1):
                for t in (-1, 1):
                    o = [0, 0, 0]
                    o[a], o[b] = s, t
                    y = y + 2 * at(*o)
    return y


@pytest.mark.parametrize("n,bc_kind", [(16, 1), (20, 2), (32, 1), (32, 2)])
def test_small_entries_beside_large_ones(n, bc_kind):
    """Two iterations from x_0 = 0 on a b of entries near 2^-10 with a 1 at every
    fourth node along each axis, so that every brick's scale is that of 1.
    x_2 = alpha_0 b + alpha_1 (b - alpha_0 A b + beta b) shows the A b of the
    first iteration entry by entry.  Bound: each tap is off by at most half
    of 2^-54 (two bits below the last place of 1), 144 in all, times alpha_0 alpha_1,
    and 64 roundings of 2^-53 of the magnitudes in the sum (about 10 on the way of an entry, the
    rest for the inner products).  Taps truncated to the last place of 1 are off by up
    to 8 times as much (4 times the bound on this data)."""
    r = np.random.Generator(np.random.PCG64(7))
    b = np.ldexp(r.uniform(0.5, 1.0, (n + 1,) * 3), -10) * r.choice([-1.0, 1.0], (n + 1,) * 3)
    b[2::4, 2::4, 2::4] = 1.0
    x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
    B.bicg_solve(B.Level(n, bc_kind), dev(b), x, 0.0, 2)
    i = slice(1, -1)
    v = b[i, i, i].astype(np.longdouble)
    q0 = _operator_ld(n, bc_kind, v)
    a0 = (v * v).sum() / (v * q0).sum()
    r1 = v - a0 * q0
    beta = (r1 * r1).sum() / (v * v).sum()
    p1 = r1 + beta * v
    a1 = (r1 * r1).sum() / (p1 * _operator_ld(n, bc_kind, p1)).sum()
    off = np.abs(x.cpu().numpy()[i, i, i] - (a0 * v + a1 * p1))
    tap, eps = np.ldexp(np.longdouble(1), -55), np.ldexp(np.longdouble(1), -53)
    bound = a0 * a1 * 144 * tap + 64 * eps * (a0 * np.abs(v) + a1 * ((1 + beta) * np.abs(v) + a0 * np.abs(q0)))
    assert float((off / bound).max()) <= 1.0


@pytest.mark.parametrize("n,bc_kind", [(54, 1), (67, 2), (81, 1)])
def test_elided_bits_with_vectors_in_shared_memory(n, bc_kind):
    """Six and eight nodes per thread keep x, r*, p* in shared memory; the elided
    form has no r*, p* there and gives the same bits."""
    b, x0 = dev(P.random_field(n, 305)), dev(P.random_field(n, 306) * 0.1)
    got = []
    for mode in ("full", "elided"):
        ctx = B.Context()
        ctx.set_shadow_mode(mode)
        x = x0.clone()
        got.append((x, B.bicg_solve(B.Level(n, bc_kind, ctx), b, x, 0.0, 40)))
    assert got[0][1] == got[1][1] and torch.equal(got[0][0], got[1][0])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_eighty_cubed_alone_and_in_a_batch(precision):
    """The largest on-chip grid of a cascade (80 = 5 * 16, eight nodes per thread), also
    as a batch member: the finest level's residual, formed again here, meets the
    tolerance (1e-3 for the two ways of forming it), and in FP64 the two agree within the
    1e-9 of a full solve."""
    n, nc, kind, tol = 80, 5, 2, 1e-8
    f, g1, g2 = (dev(a) for a in P.exp_sum().data(n, kind))
    uh = torch.empty((n + 1,) * 3, dtype=torch.float64, device=DEV)
    ut, stats = B.excmg_solve(n, nc, kind, f, g1, g2, tol, u_h_out=uh, return_stats=True, precision=precision)
    assert all(s["relres"] <= tol and not s["stagnated"] for s in stats[2:])
    lvl = B.Level(n, kind)
    fh = B.excmg_assemble_rhs(lvl, n, f, g1, g2)
    assert float((fh - B.stencil_apply(lvl, uh)).norm() / fh.norm()) <= tol * (1 + 1e-3)
    batch = B.Batch(max_instances=2)
    ids = [batch.submit(n, nc, kind, f, g1, g2, tol, precision=precision) for _ in range(2)]
    batch.run()
    for k, u in ids:
        q = batch.query(k)
        assert q["status"] == 0 and all(s["relres"] <= tol for s in q["stats"][2:])
        assert torch.equal(u, ids[0][1])
        if precision == "fp64":
            assert float((u - ut).abs().max()) <= 1e-9 * float(ut.abs().max())
