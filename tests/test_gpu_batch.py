"""The batch engine: many EXCMG solves resident on one GPU, their Bi-CG
iterations advanced per level group (one cooperative launch for small grids
and FP32 correction solves, the single solver's kernels per member on large
FP64 grids)."""
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

# (n_finest, n_coarsest, bc_kind, problem)
# first-kind random sines on 64^3 need ~1100 oracle Bi-CG iterations on the
# finest level (minutes of CPU time): the 64^3 instance has second-kind data
MIX = [(32, 4, 1, "sin_pi"), (48, 6, 2, "random_sines:3"), (64, 8, 2, "random_sines:4"),
       (24, 6, 2, "exp_sum"), (40, 5, 1, "sin2pi_plus_poly")]

_ORACLE = {}


def oracle_solution(n, nc, bc, name, tol):
    """u~ of the oracle for one MIX entry (computed once per session)."""
    key = (n, nc, bc, name, tol)
    if key not in _ORACLE:
        fr, g1r, g2r = P.by_name(name).data(n, bc)
        _ORACLE[key] = oracle.excmg(n, nc, bc, fr, g1r, g2r, tol)[1]
    return _ORACLE[key]


def data(n, bc, name):
    prob = P.by_name(name)
    f, g1, g2 = prob.data(n, bc)
    return prob, tuple(torch.from_numpy(np.array(a, order="C")).to(DEV) for a in (f, g1, g2))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_matches_single_solves_and_oracle(precision):
    """A mix of sizes, coarsest grids and kinds solved together matches each
    instance solved alone and the oracle.  FP64: within the 1e-9 bound of a
    full solve; mixed: reaches the same FP64 residual tolerance."""
    tol = 1e-10
    batch = B.Batch(max_instances=16)
    subs = []
    for n, nc, bc, name in MIX:
        prob, (f, g1, g2) = data(n, bc, name)
        ident, u = batch.submit(n, nc, bc, f, g1, g2, tol, precision=precision)
        subs.append((ident, u, n, nc, bc, prob, f, g1, g2))
    batch.run()
    for (ident, u, n, nc, bc, prob, f, g1, g2), (_, _, _, name) in zip(subs, MIX):
        q = batch.query(ident)
        assert q["done"] and q["status"] == 0
        for s in q["stats"][2:]:
            assert s["relres"] <= tol
        ref_t = oracle_solution(n, nc, bc, name, tol)
        got = u.cpu().numpy()
        scale = np.abs(ref_t).max()
        if precision == "fp64":
            single = B.excmg_solve(n, nc, bc, f, g1, g2, tol)
            assert np.abs(got - ref_t).max() <= 1e-9 * scale
            assert np.abs(got - single.cpu().numpy()).max() <= 1e-9 * scale
        else:
            disc = np.abs(ref_t - prob.exact(n)).max()
            assert np.abs(got - ref_t).max() <= 0.05 * disc


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_result_is_the_same_alone_and_in_the_mix(precision):
    """An instance's tiles, chunks and partial sums never mix with another
    instance's, so its result does not depend on what else is running --
    bit for bit."""
    n, nc, bc, name = 48, 6, 1, "random_sines:7"
    _, (f, g1, g2) = data(n, bc, name)
    alone = B.Batch(max_instances=4)
    _, ua = alone.submit(n, nc, bc, f, g1, g2, 1e-10, precision=precision)
    alone.run()
    mixed = B.Batch(max_instances=8)
    others = []
    for k, (m, mc, mb, mn) in enumerate(MIX[:3]):
        _, (mf, mg1, mg2) = data(m, mb, mn)
        others.append(mixed.submit(m, mc, mb, mf, mg1, mg2, 1e-10, precision=["fp64", "mixed"][k % 2]))
    mixed.step()
    mixed.step()           # the instance joins a batch already under way
    ident, um = mixed.submit(n, nc, bc, f, g1, g2, 1e-10, precision=precision)
    mixed.run()
    assert mixed.query(ident)["done"]
    assert torch.equal(ua, um)


def test_batch_launched_levels_match_single_solves():
    """FP64 instances whose levels above 64^3 run in launched mode (per
    member the single solver's operator and update kernels on the group's
    stream) next to small cooperative ones: every level meets the tolerance,
    results agree with each instance solved alone within the 1e-9 bound of a
    full solve, and a launched-mode instance gives the same bits alone and in
    the mix."""
    tol = 1e-10
    cases = [(96, 6, 2, "exp_sum"), (128, 8, 2, "random_sines:5"), (32, 4, 1, "sin_pi"), (64, 8, 2, "sin_pi")]
    batch = B.Batch(max_instances=8)
    subs = []
    for n, nc, bc, name in cases:
        _, (f, g1, g2) = data(n, bc, name)
        ident, u = batch.submit(n, nc, bc, f, g1, g2, tol, precision="fp64")
        subs.append((ident, u, n, nc, bc, f, g1, g2))
    batch.run()
    prof = batch.profile()
    assert prof["group_launches"] > 0 and prof["rounds"] > 0
    assert 0 < prof["member_iters"] <= prof["member_rounds"]
    for ident, u, n, nc, bc, f, g1, g2 in subs:
        q = batch.query(ident)
        assert q["done"] and q["status"] == 0
        for s in q["stats"][2:]:
            assert s["relres"] <= tol or s["stagnated"]
        single = B.excmg_solve(n, nc, bc, f, g1, g2, tol)
        scale = float(single.abs().max())
        assert float((u - single).abs().max()) <= 1e-9 * scale
    n, nc, bc, name = cases[1]
    _, (f, g1, g2) = data(n, bc, name)
    alone = B.Batch(max_instances=2)
    _, ua = alone.submit(n, nc, bc, f, g1, g2, tol, precision="fp64")
    alone.run()
    assert torch.equal(ua, subs[1][1])


def test_batch_admission_respects_the_budget():
    n, nc = 32, 4
    need = B.Batch.instance_bytes(n, nc, "mixed")
    batch = B.Batch(hbm_budget_bytes=int(need * 1.5), max_instances=8)
    _, (f, g1, g2) = data(n, 1, "sin_pi")
    first = batch.submit(n, nc, 1, f, g1, g2, 1e-10)
    assert first is not None
    assert batch.submit(n, nc, 1, f, g1, g2, 1e-10) is None     # over budget: not admitted
    batch.run()
    assert batch.query(first[0])["done"]
    assert batch.bytes == 0
    assert batch.submit(n, nc, 1, f, g1, g2, 1e-10) is not None  # room again
    batch.run()


def test_correction_solves_above_the_on_chip_grids_beside_small_requests():
    """Mixed-precision requests whose finest level takes cooperative groups beside a stream of
    small on-chip ones: all end, each level at its tolerance, and the large ones give the bits
    that they give alone."""
    tol = 1e-8
    _, big = data(96, 2, "exp_sum")
    _, small = data(32, 2, "random_sines:1")
    alone = B.Batch(max_instances=2)
    _, want = alone.submit(96, 6, 2, *big, tol, precision="mixed")
    alone.run()
    batch = B.Batch(max_instances=20)
    large = [batch.submit(96, 6, 2, *big, tol, precision="mixed") for _ in range(2)]
    live = [batch.submit(32, 4, 2, *small, tol, precision="fp64")[0] for _ in range(12)]
    done = 0
    while not all(batch.query(k)["done"] for k, _ in large) and done < 2000:
        batch.step()
        left = [k for k in live if not batch.query(k)["done"]]
        done += len(live) - len(left)
        live = left + [batch.submit(32, 4, 2, *small, tol, precision="fp64")[0] for _ in range(12 - len(left))]
    batch.run()
    for k, u in large:
        q = batch.query(k)
        assert q["done"] and q["status"] == 0
        assert all(s["relres"] <= tol for s in q["stats"][2:])
        assert torch.equal(u, want)
