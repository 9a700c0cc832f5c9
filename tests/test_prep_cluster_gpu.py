"""Small problems prepared by one cluster of blocks against the float64 oracle
(the suite's tolerances) at the edges: one row, row counts around the mean's chunks of 256 and the operand
blocks, every lane count per row, ragged widths, both sides of the size
limits, records, signs and flags."""
import numpy as np
import pytest

from oracle import oracle_sum
from paper_2609_04910_gb300.workloads import generate, to_device
from tests.gpu_helpers import TOL, case, forward_check, rel_err

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
@pytest.mark.parametrize("M,N,D,C", [(1, 1, 1, 1), (1, 2047, 3, 1), (255, 257, 16, 2), (1024, 1024, 64, 1),
                                     (1024, 1025, 64, 1), (700, 301, 100, 4), (1000, 1040, 63, 3),
                                     (300, 200, 200, 1), (511, 1, 256, 2), (257, 255, 255, 1)])
def test_single_problems(M, N, D, C, dtype):
    forward_check(case(M, N, D, C, dtype, kind="offset", tau=10.0 / D))
    forward_check(case(M, N, D, C, dtype))


@pytest.mark.parametrize("M,N,D,same", [(600, 600, 32, True), (1000, 1000, 20, False), (129, 1900, 7, False)])
def test_batches_on_both_sides_of_the_limit(M, N, D, same):
    """Up to 19 problems fit one wave of clusters, 20 take the separate
    launches."""
    import paper_2609_04910_gb300 as gs
    inp = generate(case(M, N, D, 1, "fp16", kind="mmd" if same else "normal", q_is_k=same), seed=2)
    ref, den = oracle_sum(inp["q64"], inp["k64"], inp["v64"], 1.0 / D)
    for B in (1, 3, 19, 20):
        k = torch.stack([to_device(inp["k"], "fp16")] * B).contiguous()
        q = k if same else torch.stack([to_device(inp["q"], "fp16")] * B).contiguous()
        v = torch.stack([to_device(inp["v"], "fp16")] * B).contiguous()
        got = gs.gauss_sum_batched(q, k, v, 1.0 / D)
        gs.gauss_sum_device_status()
        for b in range(B):
            assert rel_err(got[b].cpu().numpy(), ref, den) <= TOL["fp16"]


@pytest.mark.parametrize("N,D,dtype", [(2048, 16, "fp16"), (2049, 16, "fp16"), (1000, 50, "fp16"),
                                       (600, 32, "bf16")])
@pytest.mark.parametrize("B", [1, 4])
def test_mmd2_with_signs_and_flags(N, D, dtype, B):
    import paper_2609_04910_gb300 as gs
    inp = [generate(case(N, N, D, 1, dtype, kind="mmd", q_is_k=True), seed=s) for s in range(B)]
    x = torch.stack([to_device(i["k"], dtype) for i in inp]).contiguous()
    v = torch.stack([to_device(i["v"], dtype) for i in inp])[..., 0].contiguous()
    got = gs.gauss_sum_mmd2(x, v, 1.0 / D).cpu().numpy()
    gs.gauss_sum_device_status()
    for b, i in enumerate(inp):
        ref, den = oracle_sum(i["q64"], i["k64"], i["v64"], 1.0 / D)
        want = float((i["v64"][:, 0] * ref[:, 0]).sum())
        scale = float((np.abs(i["v64"][:, 0]) * den[:, 0]).sum())
        assert abs(got[b] - want) <= TOL[dtype] * scale
