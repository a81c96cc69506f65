"""The transpose and the padded copy where their tiling can go wrong: sides
around the 512-bit tile, odd word counts (rows of X and of its transpose then
start at odd 8-byte places), long thin shapes; k / 64 odd, so that the padded
copy of A and the zero words behind B^T are read, with rows shorter and longer
than the words a CTA copies."""
import numpy as np
import pytest

import oracle as O
from gpu_util import first_mismatch, from_dev, gen, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

import paper_1909_01554_gb300 as bmm  # noqa: E402


@pytest.mark.parametrize("rows,cols", [(64, 64), (448, 512), (512, 576), (576, 448), (1024, 64), (64, 1088),
                                       (960, 4160), (20032, 192), (128, 20032)])
def test_transpose_at_tile_edges(rows, cols):
    X = gen(rows, cols, 71, 0)
    T = torch.full((rows * cols // 64 + 8,), -1, dtype=torch.int64, device="cuda")
    bmm.transpose(to_dev(X), T, rows, cols)
    T = T.cpu().numpy().view(np.uint64)
    assert (T[-8:] == np.uint64(0xFFFFFFFFFFFFFFFF)).all()  # nothing behind the result
    assert first_mismatch(T[:-8].reshape(cols, rows // 64), O.transpose(X, rows, cols)) is None


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("m,k,n", [(64, 64, 64), (640, 448, 576), (4160, 192, 64), (64, 140992, 128)])
@pytest.mark.parametrize("batched", [False, True])
def test_odd_word_counts_are_padded(op, m, k, n, batched):
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, B = gen(m, k, 72, 0, p=p), gen(k, n, 72, 1, p=p)
    dA, dB, C = to_dev(A), to_dev(B), bmm.empty(m, n)
    C.fill_(-1)
    if batched:
        plan = bmm.BatchedPlan([op], [dA], [dB], [C], [m], [k], [n], path=bmm.PATH_TC_FP4_PAIR)
        plan.run()
    else:
        bmm.product(op, dA, dB, C, m, k, n, path=bmm.PATH_TC_FP4_PAIR)
    bmm.stream_status()
    assert first_mismatch(from_dev(C, m, n), O.cubic(op, A, B, m, k, n)) is None


def test_rows_too_long_for_32_bit_offsets():
    """64 rows of 2^20 + 1 words: a tile's words lie 4 GiB apart."""
    rows, words = 64, (1 << 20) + 1
    gen_ = torch.Generator(device="cuda")
    gen_.manual_seed(73)
    X = torch.randint(-2**62, 2**62, (rows * words,), dtype=torch.int64, device="cuda", generator=gen_)
    T = torch.empty_like(X)
    bmm.transpose(X, T, rows, 64 * words)
    shift = torch.arange(64, device="cuda")
    for b in range(0, 64, 7):  # bit b of every word of X: columns 64 w + b
        bits = (X.reshape(rows, words) >> b) & 1
        want = (bits << shift[:, None]).sum(0)
        assert torch.equal(T.reshape(words, 64)[:, b], want)


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
def test_batch_at_its_tile_edges(op):
    """A batch's tiles are 256 rows of B high and 512 columns wide."""
    sizes = [(64, 192, 448), (128, 256, 512), (64, 320, 576), (1088, 512, 64), (64, 576, 1088)]
    p = [None if op == bmm.GF2 else f"1/sqrt({k})" for m, k, n in sizes]
    A = [gen(m, k, 74, 2 * i, p=p[i]) for i, (m, k, n) in enumerate(sizes)]
    B = [gen(k, n, 74, 2 * i + 1, p=p[i]) for i, (m, k, n) in enumerate(sizes)]
    C = [bmm.empty(m, n) for m, k, n in sizes]
    for c in C:
        c.fill_(-1)
    dA, dB = [to_dev(x) for x in A], [to_dev(x) for x in B]
    plan = bmm.BatchedPlan([op] * len(sizes), dA, dB, C, *(list(x) for x in zip(*sizes)),
                           path=bmm.PATH_TC_FP4_PAIR)
    plan.run()
    bmm.stream_status()
    for i, (m, k, n) in enumerate(sizes):
        assert first_mismatch(from_dev(C[i], m, n), O.cubic(op, A[i], B[i], m, k, n)) is None
