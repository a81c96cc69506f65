"""Kernels that start before their predecessor has ended: chains of calls on one
stream in which every call reads what the one before wrote, and overwrites what
the one before read, through every form of product, against the same chain with
a synchronisation after every call."""
import pytest

from gpu_util import gen, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

import paper_1909_01554_gb300 as bmm  # noqa: E402

FORMS = {
    "library": {},  # one launch at 640, the tensor kernel at 2048
    "popc": {"path": bmm.PATH_POPC, "depth": 0},
    "merged levels": {"depth": 2},
    "a level at a time": {"depth": 2, "serial": 2},
    "in-kernel level": {"depth": 2, "path": bmm.PATH_POPC, "kernel_level": 1},
}


@pytest.mark.parametrize("side", [640, 2048])
@pytest.mark.parametrize("form", FORMS)
def test_every_call_reads_the_one_before(side, form):
    kw = FORMS[form]
    if kw.get("depth") and side == 640:
        kw = {**kw, "depth": 1, **({"serial": 1} if "serial" in kw else {})}
    start, M = to_dev(gen(side, side, 51, 0)), to_dev(gen(side, side, 51, 1))

    def chain(sync):
        X, Y, Z = start.clone(), torch.empty_like(start), torch.empty_like(start)
        out = []
        for i in range(24):
            bmm.gf2(X, M, Y, side, side, side, **kw)
            if sync:
                torch.cuda.synchronize()
            bmm.transpose(Y, Z, side, side)
            if sync:
                torch.cuda.synchronize()
            bmm.gf2(M, Z, X, side, side, side, **kw)
            if sync:
                torch.cuda.synchronize()
            if i % 6 == 5:
                out.append(X.clone())
        return out

    want = chain(True)
    for _ in range(5):
        got = chain(False)
        assert all(torch.equal(g, w) for g, w in zip(got, want))
    bmm.stream_status()


@pytest.mark.parametrize("variant", [bmm.SELF_INVERSE, bmm.CHAINING])
def test_basis_changes_in_place(variant):
    """Levels of one call and the calls around it, all on one buffer."""
    side, depth = 2048, 3
    start, M = to_dev(gen(side, side, 53, 0)), to_dev(gen(side, side, 53, 1))

    def chain(sync):
        X, Y = start.clone(), torch.empty_like(start)
        out = []
        for i in range(24):
            bmm.basis_change(variant, i & 1, X, side, side, depth)
            if sync:
                torch.cuda.synchronize()
            bmm.gf2(X, M, Y, side, side, side, depth=1, variant=variant)
            if sync:
                torch.cuda.synchronize()
            bmm.basis_change(variant, 1 - (i & 1), Y, side, side, depth)
            if sync:
                torch.cuda.synchronize()
            bmm.transpose(Y, X, side, side)
            if sync:
                torch.cuda.synchronize()
            if i % 6 == 5:
                out.append(X.clone())
        return out

    want = chain(True)
    for _ in range(5):
        assert all(torch.equal(g, w) for g, w in zip(chain(False), want))
    bmm.stream_status()


def test_plan_runs_back_to_back():
    """A plan over its own results: each run's outputs are the next run's inputs."""
    side, count = 448, 6
    M = to_dev(gen(side, side, 52, 1))
    bufs = [[to_dev(gen(side, side, 52, 2 + i)) for i in range(count)], [bmm.empty(side, side) for _ in range(count)]]
    plans = [bmm.BatchedPlan(bmm.GF2, bufs[a], [M] * count, bufs[1 - a], [side] * count, [side] * count, [side] * count)
             for a in (0, 1)]
    first = [b.clone() for b in bufs[0]]

    def chain(sync):
        for b, f in zip(bufs[0], first):
            b.copy_(f)
        for i in range(20):
            plans[i % 2].run()
            if sync:
                torch.cuda.synchronize()
        return [b.clone() for b in bufs[0]]

    want = chain(True)
    for _ in range(5):
        assert all(torch.equal(g, w) for g, w in zip(chain(False), want))
    bmm.stream_status()
