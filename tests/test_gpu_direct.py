"""The one-launch product of small matrices: one and several steps of k, k that
ends inside a step, k / 64 odd, k split over clusters of 2, 4 and 8 CTAs with
slices that come out uneven or empty, single and many tiles."""
import pytest

import oracle as O
from gpu_util import first_mismatch, from_dev, gen, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

import paper_1909_01554_gb300 as bmm  # noqa: E402

if not bmm.device_supported():  # pragma: no cover - other GPU
    pytest.skip("chosen on sm_103 only", allow_module_level=True)


@pytest.mark.parametrize("op", [bmm.GF2, bmm.BOOL])
@pytest.mark.parametrize("m,k,n", [(64, 64, 64), (128, 192, 64), (64, 2048, 192), (64, 2112, 64), (192, 4160, 128),
                                   (64, 8384, 64), (128, 10304, 64), (64, 12352, 64), (1024, 1024, 1024),
                                   (64, 64, 32768), (16384, 128, 64), (576, 1088, 704)])
def test_direct_matches_oracle(op, m, k, n):
    p = None if op == bmm.GF2 else f"1/sqrt({k})"
    A, B = gen(m, k, 61, 0, p=p), gen(k, n, 61, 1, p=p)
    dA, dB, want = to_dev(A), to_dev(B), O.cubic(op, A, B, m, k, n)
    C = torch.full((m * n // 64 + 8,), -1, dtype=torch.int64, device="cuda")
    for _ in range(3):
        l0 = bmm.launch_count()
        bmm.product(op, dA, dB, C, m, k, n)
        assert bmm.launch_count() == l0 + 1  # this form, not transpose and product
        bmm.stream_status()
        assert first_mismatch(from_dev(C[:-8], m, n), want) is None
    assert int((C[-8:] != -1).sum()) == 0  # nothing behind the result


def test_explicit_paths_and_workspaces_keep_the_general_form():
    m, k, n = 256, 512, 384
    A, B = gen(m, k, 62, 0), gen(k, n, 62, 1)
    dA, dB, want = to_dev(A), to_dev(B), O.cubic(O.GF2, A, B, m, k, n)
    for path in (bmm.PATH_POPC, *bmm.TENSOR_PATHS):
        C = bmm.empty(m, n)
        l0 = bmm.launch_count()
        bmm.gf2(dA, dB, C, m, k, n, path=path)
        assert bmm.launch_count() == l0 + 2
        assert first_mismatch(from_dev(C, m, n), want) is None
    size = bmm.workspace_size(bmm.GF2, m, k, n)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    C = bmm.empty(m, n)
    bmm.gf2(dA, dB, C, m, k, n, workspace=ws, workspace_bytes=size)
    assert first_mismatch(from_dev(C, m, n), want) is None
    with pytest.raises(bmm.BmmError):
        bmm.gf2(dA, dB, C, m, k, n, workspace=ws, workspace_bytes=size - 1)
