"""Sums with the query rows in tensor memory (16-bit rows too wide for the
augmented layout, guarded fp32 sums of 33 to 64 coordinates): one warp issues
all MMAs of a block and S tiles go back to it tile by tile.  Long and ragged
key ranges, several segments per block, every channel count: repeated calls
agree bit for bit and sampled rows agree with the float64 oracle to the
suite's tolerances."""
import numpy as np
import pytest

from oracle import oracle_sum
from paper_2609_04910_gb300.workloads import device_inputs, generate
from tests.gpu_helpers import TOL, case, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


# (M x N: one segment per block over many key tiles, segments that end inside
# a pair of query tiles, many short segments per block, one key tile each.)
@pytest.mark.parametrize("dtype,D,C", [("fp32", 33, 1), ("fp32", 41, 2), ("fp32", 57, 3), ("fp32", 64, 4),
                                       ("fp32", 64, 1), ("fp16", 125, 1), ("fp16", 256, 4),
                                       ("bf16", 131, 2), ("bf16", 200, 3)])
@pytest.mark.parametrize("M,N", [(16384, 16384), (20000, 17001), (2500, 70001), (40000, 450), (70000, 256)])
def test_repeats_and_sampled_rows(dtype, D, C, M, N):
    import paper_2609_04910_gb300 as gs
    inp = generate(case(M, N, D, C, dtype), seed=8)
    q, k, v = device_inputs(inp)
    first = gs.gauss_sum(q, k, v, 1.0 / D)
    again = [gs.gauss_sum(q, k, v, 1.0 / D) for _ in range(12)]
    gs.gauss_sum_device_status()
    assert all(torch.equal(first, a) for a in again)
    rows = np.unique(np.concatenate([np.arange(0, M, M // 24), np.arange(M - 3, M)]))
    ref, den = oracle_sum(inp["q64"], inp["k64"], inp["v64"], 1.0 / D, rows=rows)
    assert rel_err(first.cpu().numpy()[rows], ref, den) <= TOL[dtype]
