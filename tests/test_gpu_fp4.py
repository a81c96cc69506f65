"""The e2m1 tensor kernel where its tiling can go wrong: k that ends inside a
384-bit stage, a stage ring that wraps, column tiles of 64 to 256 columns, row
tiles cut short, several tiles per CTA pair. Small shapes against the CPU
oracle; large ones, many times over, against the e4m3 kernel (bit for bit)."""
import pytest

import oracle as O
from gpu_util import first_mismatch, from_dev, gen, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

import paper_1909_01554_gb300 as bmm  # noqa: E402

if not bmm.device_supported():  # pragma: no cover - other GPU
    pytest.skip("tensor-core paths need sm_103", allow_module_level=True)

FP4 = bmm.PATH_TC_FP4_PAIR


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("k", [128, 256, 384, 512, 768, 896, 1152, 1536, 3072, 3200, 6272])
def test_k_ends_anywhere_in_a_stage(op, k):
    m, n = 320, 448
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, B = gen(m, k, 81, 0, p=p), gen(k, n, 81, 1, p=p)
    C = bmm.empty(m, n)
    C.fill_(-1)
    bmm.product(op, to_dev(A), to_dev(B), C, m, k, n, path=FP4, **({"depth": 0} if op == bmm.GF2 else {}))
    bmm.stream_status()
    assert first_mismatch(from_dev(C, m, n), O.cubic(op, A, B, m, k, n)) is None


@pytest.mark.parametrize("m", [64, 128, 192, 256, 320])
@pytest.mark.parametrize("n", [64, 128, 192, 256, 320, 384])
def test_ragged_tiles(m, n):
    k = 1024
    A, B = gen(m, k, 82, 0), gen(k, n, 82, 1)
    C = bmm.empty(m, n)
    C.fill_(-1)
    bmm.gf2(to_dev(A), to_dev(B), C, m, k, n, path=FP4, depth=0)
    bmm.stream_status()
    assert first_mismatch(from_dev(C, m, n), O.cubic(O.GF2, A, B, m, k, n)) is None


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("m,k,n", [(64, 1536, 64),       # one tile, a stage a slice
                                   (320, 9984, 448),     # four tiles, 26 stages in 13 slices
                                   (512, 12352, 320),    # k / 64 odd, uneven last slice
                                   (256, 33344, 9728),   # 38 tiles, two slices each
                                   (2112, 1984, 2240),   # a round of whole tiles, then five of six slices
                                   (10240, 1600, 2496),  # five rounds, twenty tiles of three slices, the
                                                         # last column of tiles narrow
                                   (1088, 66048, 128)])  # slices longer than a Boolean segment
def test_slices_of_k(op, m, k, n):
    """Tiles cut along k, combined into C: what C held before, and what the call
    before left there, must not show."""
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, B = to_dev(gen(m, k, 84, 0, p=p)), to_dev(gen(k, n, 84, 1, p=p))
    kw = {"depth": 0} if op == bmm.GF2 else {}
    want = bmm.empty(m, n)
    bmm.product(op, A, B, want, m, k, n, path=bmm.PATH_POPC, **kw)
    C = torch.full((m * n // 64 + 8,), -1, dtype=torch.int64, device="cuda")
    for _ in range(20):
        bmm.product(op, A, B, C, m, k, n, path=FP4, **kw)
        assert torch.equal(C[:-8], want) and int((C[-8:] != -1).sum()) == 0
    bmm.stream_status()


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("k", [32640, 32768, 32896, 65280, 65408, 98432])
def test_counts_around_the_flushes(op, k):
    """Prefix rows: entry (i, j) of the integer product is min(a_i, b_j), which
    takes every count at the ends of the segments that Boolean counts are
    accumulated in (2^15), 0 and k among them."""
    m, n = 256, 320
    edges = [0, 1, 2, 127, 255, 256, 32639, 32640, 32641, 32767, 32768, 32769, 65279, 65280, 65281, k - 1, k]
    a = [min(edges[i % len(edges)], k) if i < 128 else (i * 7919) % (k + 1) for i in range(m)]
    b = [min(edges[(i // 3) % len(edges)], k) if i < 160 else k - (i * 104729) % (k + 1) for i in range(n)]

    def prefix(counts):
        w = torch.zeros((len(counts), k // 64), dtype=torch.int64)
        for i, c in enumerate(counts):
            w[i, : c // 64] = -1
            if c % 64:
                w[i, c // 64] = (1 << (c % 64)) - 1
        return w.reshape(-1).cuda()

    C = bmm.empty(m, n)
    C.fill_(-1)
    bmm.base_product(op, FP4, prefix(a), prefix(b), C, m, k, n)
    bmm.stream_status()
    count = torch.minimum(torch.tensor(a)[:, None], torch.tensor(b)[None, :])
    want = count % 2 if op == bmm.GF2 else (count > 0).to(torch.int64)
    got = (C.cpu().reshape(m, n // 64, 1) >> torch.arange(64)) & 1
    assert torch.equal(got.reshape(m, n), want)


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("m,k,n,runs", [(4096, 4096, 4096, 100), (8192, 384, 8192, 50), (8192, 128, 8256, 50),
                                        (4096, 16384, 4224, 10)])
def test_many_tiles_many_times(op, m, k, n, runs):
    """Every word of every run: an operand read before it is complete, or after
    the next copy has overwritten it, shows as a few wrong words in one run."""
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, Bt = to_dev(gen(m, k, 83, 0, p=p)), to_dev(gen(n, k, 83, 1, p=p))
    want, C = bmm.empty(m, n), bmm.empty(m, n)
    bmm.base_product(op, bmm.PATH_TC_FP8_PAIR, A, Bt, want, m, k, n)
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(runs):
        bmm.base_product(op, FP4, A, Bt, C, m, k, n)
        wrong += (C != want).sum()
    bmm.stream_status()
    assert int(wrong) == 0
