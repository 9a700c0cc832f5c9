"""Vectorised preparation (common mean, operand rows) for widths that are no
multiple of 8: odd, even and multiple-of-4 D on one, two and four lanes per
row, augmented and plain layouts, q = k, batches whose problems start off a
16-byte boundary, against the float64 oracle (the suite's tolerances).  The
clouds share an offset of norm 50, so that a wrong mean shows."""
import numpy as np
import pytest

from oracle import oracle_sum
from paper_2609_04910_gb300.workloads import generate, to_device
from tests.gpu_helpers import TOL, case, forward_check, grad_check, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("D", [1, 2, 3, 7, 9, 12, 20, 50, 63, 65, 77, 100, 121, 124, 125, 129, 200,
                               201, 255])
def test_offset_clouds(D, dtype):
    # tau as in the offset workload; bf16 spacing at coordinates of 50 / sqrt(D)
    # is coarse, but the oracle sees the same rounded points.
    forward_check(case(1500, 2111, D, 1, dtype, kind="offset", tau=10.0 / D))
    forward_check(case(131, 1025, D, 2, dtype, kind="offset", tau=10.0 / D))


@pytest.mark.parametrize("D", [3, 20, 50, 100])
def test_q_is_k_and_gradient(D):
    forward_check(case(1111, 1111, D, 1, "fp16", kind="mmd", q_is_k=True))
    grad_check(case(1111, 1111, D, 1, "fp16", kind="gmm", q_is_k=True))
    grad_check(case(300, 2049, D, 1, "bf16"))


@pytest.mark.parametrize("M,N,D", [(5, 1031, 3), (1030, 1100, 9), (1001, 1003, 50), (1024, 1024, 12)])
def test_batches_off_the_vector_boundary(M, N, D):
    import paper_2609_04910_gb300 as gs
    B = 3
    inp = [generate(case(M, N, D, 1, "fp16"), seed=s) for s in range(B)]
    q, k, v = (torch.stack([to_device(i[n], "fp16") for i in inp]).contiguous() for n in "qkv")
    got = gs.gauss_sum_batched(q, k, v, 1.0 / D).cpu().numpy()
    gs.gauss_sum_device_status()
    for b, i in enumerate(inp):
        ref, den = oracle_sum(i["q64"], i["k64"], i["v64"], 1.0 / D)
        assert rel_err(got[b], ref, den) <= TOL["fp16"]
