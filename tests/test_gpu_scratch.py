"""Scratch and buffers kept between calls: products from several threads and
streams at once, after the kept memory has been given back, and host-memory
products of changing shapes under a device budget."""
import threading

import numpy as np
import pytest

import oracle as O
from gpu_util import first_mismatch, from_dev, gen, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

import paper_1909_01554_gb300 as bmm  # noqa: E402


def test_threads_and_streams_share_the_pool():
    """Forms that take scratch, of different sizes, so that a block freed on one
    stream is taken again on another."""
    shapes = [(1024, 1088, 960, {"path": bmm.PATH_TC_FP4_PAIR, "depth": 0}),  # k / 64 odd: A padded too
              (192, 2112, 256, {"path": bmm.PATH_TC_FP4_PAIR, "depth": 0}),
              (512, 1024, 640, {"path": bmm.PATH_POPC, "depth": 0}),
              (2048, 1024, 1536, {"depth": 1})]
    if not bmm.device_supported():  # pragma: no cover - other GPU
        shapes = [(m, k, n, {**kw, "path": bmm.PATH_POPC}) for m, k, n, kw in shapes]
    assert len({bmm.workspace_size(bmm.GF2, m, k, n, **kw) for m, k, n, kw in shapes}) == len(shapes)
    jobs = []
    for t, (m, k, n, kw) in enumerate(shapes):
        A, B = gen(m, k, 91 + t, 0), gen(k, n, 91 + t, 1)
        jobs.append((m, k, n, kw, to_dev(A), to_dev(B), [bmm.empty(m, n) for _ in range(20)],
                     O.cubic(O.GF2, A, B, m, k, n)))
    torch.cuda.synchronize()
    errors = []
    before = bmm.launch_count()

    def work(job):
        m, k, n, kw, dA, dB, Cs, _ = job
        try:
            s = torch.cuda.Stream()
            for C in Cs:
                bmm.gf2(dA, dB, C, m, k, n, stream=s, **kw)
            s.synchronize()
        except Exception as e:  # pragma: no cover - reported below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    # two launches a cubic call and four at depth 1: none took the form without scratch
    assert bmm.launch_count() - before == 20 * (2 + 2 + 2 + 4)
    bmm.stream_status()
    for m, k, n, _, _, _, Cs, want in jobs:
        for C in Cs:
            assert first_mismatch(from_dev(C, m, n), want) is None


def test_scratch_is_given_back_and_taken_again():
    m = k = n = 8192
    A, B = to_dev(gen(m, k, 95, 0)), to_dev(gen(k, n, 95, 1))
    C, D = bmm.empty(m, n), bmm.empty(m, n)
    bmm.gf2(A, B, C, m, k, n, depth=1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    bmm.host_release()
    assert torch.cuda.mem_get_info()[0] > before
    bmm.gf2(A, B, D, m, k, n, depth=2)
    bmm.stream_status()
    assert torch.equal(C, D)


@pytest.mark.parametrize("budget", [(8 << 20) + (3 << 18), 1 << 30])
def test_host_products_of_changing_shapes(budget):
    """One cache serves shapes that grow and shrink, blocked or whole."""
    bmm.host_release()
    for i, (op, m, k, n) in enumerate([(bmm.GF2, 512, 1024, 768), (bmm.BOOL, 1024, 640, 512),
                                       (bmm.GF2, 256, 512, 320), (bmm.GF2, 1536, 1024, 1024),
                                       (bmm.GF2, 512, 1024, 768)]):
        p = None if op == bmm.GF2 else f"1/sqrt({k})"
        A, B = gen(m, k, 97 + i, 0, p=p), gen(k, n, 97 + i, 1, p=p)
        C = np.full((m, n // 64), 0xFFFFFFFFFFFFFFFF, dtype=np.uint64)
        bmm.product_host(op, A, B, C, m, k, n, device_bytes=budget, host_depth=0)
        assert first_mismatch(C, O.cubic(op, A, B, m, k, n)) is None


def test_idle_scratch_is_room_for_plans_and_host_products():
    """On a device that is nearly full, what the pool keeps between calls is
    still there for the library's other allocations."""
    m = 16384
    A, B = to_dev(gen(m, m, 101, 0)), to_dev(gen(m, m, 101, 1))
    C, D = bmm.empty(m, m), bmm.empty(m, m)
    Ah, Bh, Ch = A.cpu(), B.cpu(), torch.empty(m * m // 64, dtype=torch.int64)
    warm = bmm.BatchedPlan([bmm.BOOL], [A], [B], [D], [m], [m], [m], path=bmm.PATH_POPC)  # (measures the model)
    warm.destroy()
    bmm.host_release()
    torch.cuda.empty_cache()
    bmm.gf2(A, B, C, m, m, m, depth=2, serial=0)  # about 330 MiB of scratch, kept idle
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < 310 << 20
        plan = bmm.BatchedPlan([bmm.BOOL] * 14, [A] * 14, [B] * 14, [D] * 14, [m] * 14, [m] * 14, [m] * 14,
                               path=bmm.PATH_POPC)  # 14 transposes: 448 MiB
        plan.destroy()
        bmm.gf2(A, B, C, m, m, m, depth=2, serial=0)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] < 310 << 20
        # about 400 MiB at once, half of it without the idle bytes
        assert bmm.host_plan(bmm.GF2, m, m, m)["count"] == 1
        bmm.product_host(bmm.GF2, Ah, Bh, Ch, m, m, m)
        assert torch.equal(Ch, C.cpu())
    finally:
        del hog
        bmm.host_release()
        torch.cuda.empty_cache()
