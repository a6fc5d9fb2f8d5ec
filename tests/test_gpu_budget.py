"""Under a device-memory budget a call takes the same path, and gives the same
bits, as without one and whatever the context did before: the exchange words of
the on-chip kernels lie in memory that the call's vectors need in any case."""
import numpy as np
import pytest

from paper_1901_05118_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1901_05118_gb300 import binding as B  # noqa: E402

DEV = torch.device("cuda", 0)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def least_budget(call, low, high, step=1 << 14):
    """The least budget (to `step`) with which call(budget) is not refused."""
    while high - low > step:
        mid = (low + high) // 2
        try:
            call(mid)
            high = mid
        except B.ExcmgError as e:
            assert e.status == -9
            low = mid
    return high


@pytest.mark.parametrize("n", [16, 48, 72])
def test_six_vectors_are_room_for_both_modes(n):
    """The full mode's six vectors are all that it and the elided mode need up to 81^3."""
    b = dev(P.random_field(n, 501))
    got = {}
    for mode in ("full", "elided"):
        for budget in (0, 6 * 8 * (n + 1) ** 3):
            ctx = B.Context(hbm_budget_bytes=budget)
            ctx.set_shadow_mode(mode)
            x = torch.zeros((n + 1,) * 3, dtype=torch.float64, device=DEV)
            it, rel, _ = B.bicg_solve(B.Level(n, 2, ctx), b, x, 0.0, 25)
            assert not budget or ctx.bytes <= budget
            got[mode, budget] = (x, it, rel)
    x0, it0, rel0 = got["full", 0]
    for x, it, rel in got.values():
        assert (it, rel) == (it0, rel0) and torch.equal(x, x0)


@pytest.mark.parametrize("n,nc,kind", [(48, 6, 1), (128, 8, 2)])
@pytest.mark.parametrize("mode", ["full", "elided"])
def test_repeated_solves_under_the_least_budget(n, nc, kind, mode):
    data = [dev(a) for a in P.exp_sum().data(n, kind)]

    def solve(budget, times=1):
        ctx = B.Context(hbm_budget_bytes=budget)
        ctx.set_shadow_mode(mode)
        out = [B.excmg_solve(n, nc, kind, *data, 1e-10, ctx=ctx) for _ in range(times)]
        assert not budget or ctx.bytes <= budget
        return out

    want = solve(0)[0]
    least = least_budget(solve, 1 << 14, 20 * 8 * (n + 1) ** 3 + (1 << 25))
    for got in solve(least, times=3):
        assert torch.equal(got, want)


@pytest.mark.parametrize("n", [97, 512, 600])
def test_2d_bicg_in_seven_vectors(n):
    """The 2D call's right-hand side and six vectors are all that it needs."""
    b = dev(P.random_field_2d(n, 502))
    got = []
    for budget in (0, 7 * 8 * (n + 1) ** 2):
        ctx = B.Context(hbm_budget_bytes=budget)
        for _ in range(2):
            x = torch.zeros((n + 1,) * 2, dtype=torch.float64, device=DEV)
            got.append((x, B.bicg_solve2d(n, 1, b, x, 0.0, 25, ctx=ctx)))
    for x, info in got:
        assert info == got[0][1] and torch.equal(x, got[0][0])


def test_2d_solves_under_the_least_budget():
    n, nc, kind = 128, 8, 2
    data = [dev(a) for a in P.exp_sum_2d().data(n, kind)]

    def solve(budget, times=1):
        ctx = B.Context(hbm_budget_bytes=budget)
        return [B.excmg_solve2d(n, nc, kind, *data, 1e-8, ctx=ctx) for _ in range(times)]

    want = solve(0)[0]
    for got in solve(least_budget(solve, 1 << 14, 20 * 8 * (n + 1) ** 2 + (1 << 25)), times=3):
        assert torch.equal(got, want)


@pytest.mark.parametrize("n,nc,kind", [(48, 6, 1), (80, 5, 2), (96, 6, 2)])
def test_mixed_solves_under_the_least_budget(n, nc, kind):
    """FP32 correction solves on chip up to 81^3, launched above."""
    data = [dev(a) for a in P.exp_sum().data(n, kind)]

    def solve(budget, times=1):
        ctx = B.Context(hbm_budget_bytes=budget)
        return [B.excmg_solve(n, nc, kind, *data, 1e-8, ctx=ctx, precision="mixed") for _ in range(times)]

    want = solve(0)[0]
    for got in solve(least_budget(solve, 1 << 14, 20 * 8 * (n + 1) ** 3 + (1 << 25)), times=3):
        assert torch.equal(got, want)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_levels_on_chip_take_no_memory_beyond_the_instances(precision):
    """Once its group records exist, a batch whose levels run on chip holds what its instances
    were admitted with (free memory is counted in steps of up to 2 MB)."""
    n, nc, kind = 80, 5, 2
    big, small = ([dev(a) for a in P.exp_sum().data(m, kind)] for m in (n, 20))
    batch = B.Batch(max_instances=8)
    for _ in range(4):   # the records and the direct solves' tables
        batch.submit(20, nc, kind, *small, 1e-8, precision=precision)
    batch.run()
    ids = [batch.submit(n, nc, kind, *big, 1e-8, precision=precision)[0] for _ in range(4)]
    torch.cuda.synchronize()
    before = least = torch.cuda.mem_get_info()[0]
    while not all(batch.query(k)["done"] for k in ids):
        batch.step()
        least = min(least, torch.cuda.mem_get_info()[0])
    assert before - least <= 2 << 20
    assert all(batch.query(k)["status"] == 0 for k in ids)
    batch.close()
