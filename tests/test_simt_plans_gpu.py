"""fp32 sums on the SIMT kernel where its plan changes: few rows against many
keys (blocks of 32 and 64 threads, hundreds of key splits whose partial sums
are added by several threads per output), few keys, and both sides of the
number of splits at which the additions change.  Against the float64 oracle
with the suite's tolerance; repeated calls agree bit for bit."""
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


def _check(M, N, D, C, **kw):
    import paper_2609_04910_gb300 as gs
    inp = generate(case(M, N, D, C, "fp32"), seed=31)
    q, k, v = device_inputs(inp)
    got = gs.gauss_sum(q, k, v, 1.0 / D, path=gs.GS_PATH_SIMT, **kw)
    assert torch.equal(got, gs.gauss_sum(q, k, v, 1.0 / D, path=gs.GS_PATH_SIMT, **kw))
    rows = np.unique(np.append(np.arange(0, M, max(1, M // 40)), M - 1))
    ref, den = oracle_sum(inp["q64"], inp["k64"], inp["v64"], 1.0 / D, rows=rows)
    assert rel_err(got.cpu().numpy()[rows], ref, den) <= TOL["fp32"]


@pytest.mark.parametrize("M,N", [(1, 65537), (31, 20001), (33, 70000), (129, 30000), (513, 8192),
                                 (3000, 3001), (70000, 33), (5, 7)])
@pytest.mark.parametrize("D,C", [(3, 1), (16, 4), (32, 5), (33, 2), (49, 1), (56, 4), (57, 2), (64, 3), (100, 1), (128, 4)])
def test_shapes(M, N, D, C):
    _check(M, N, D, C)


@pytest.mark.parametrize("splits", [1, 2, 3, 4, 5, 15, 16, 17, 24, 63, 64, 65, 200])
@pytest.mark.parametrize("M,C", [(1, 1), (31, 3), (257, 4)])
def test_splits(splits, M, C):
    _check(M, 6400, 20, C, split_n=splits)


@pytest.mark.parametrize("N", [7093, 7094, 8191, 8192])
@pytest.mark.parametrize("D", [2, 4])
def test_workspace_serves_one_cloud_and_two(N, D):
    """Sums of one cloud with itself change paths at another size than sums of
    two clouds; the workspace asked for holds either."""
    import paper_2609_04910_gb300 as gs
    inp = generate(case(N, N, D, 1, "fp32"), seed=32)
    q, k, v = device_inputs(inp)
    ws = torch.empty(gs.gauss_sum_workspace_size(N, N, D, 1, gs.GS_FP32), dtype=torch.uint8, device="cuda")
    for a in (k, q):
        assert torch.equal(gs.gauss_sum(a, k, v, 1.0 / D, workspace=ws), gs.gauss_sum(a, k, v, 1.0 / D))
        gs.gauss_sum_noalloc(a, k, v, 1.0 / D)
