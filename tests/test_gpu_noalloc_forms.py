"""The forms of the allocation-free product: one launch without scratch, the
tensor kernel on B^T alone, on B^T and a padded A that just fit the fixed array,
and the CUDA-core kernel where k / 64 is odd and the padded A does not fit."""
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

ARRAY = 8 << 20


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("m,k,n", [(256, 512, 384),       # one launch
                                   (1920, 2048, 2112),    # tensor, B^T alone
                                   (1088, 8192, 8192),    # B^T fills the array
                                   (12864, 2624, 12096),  # k / 64 odd: padded A and B^T fill all but 2 KiB
                                   (12928, 2624, 12096)])  # 64 rows more: A as it is, CUDA cores
def test_every_form_twice(op, m, k, n):
    kp = (k + 127) // 128 * 128
    assert n * kp // 8 <= ARRAY
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, C, want = to_dev(gen(m, k, 63, 0, p=p)), bmm.empty(m, n), bmm.empty(m, n)
    for i in range(2):  # the second call finds the first one's words in the array
        Bh = gen(k, n, 63, 1 + i, p=p)
        B = to_dev(Bh)
        C.fill_(-1)
        bmm.product_noalloc(op, A, B, C, m, k, n)
        bmm.stream_status()
        bmm.product(op, A, B, want, m, k, n, path=bmm.PATH_POPC, **({"depth": 0} if op == bmm.GF2 else {}))
        assert torch.equal(C, want)
    if m * k * n < 1 << 28:
        assert first_mismatch(from_dev(C, m, n), O.cubic(op, A.cpu().numpy().view("uint64").reshape(m, k // 64), Bh, m, k, n)) is None
