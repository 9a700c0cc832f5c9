"""Value channels of the gradient passes on both sides of the switch from blocks
of 32 rows to blocks of 128 (163840 keys, 98304 below 32 coordinates), and at
the edges of a block, against the float64 oracle with the suite's tolerances."""
import numpy as np
import pytest

from tests.gpu_helpers import case, grad_check

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
@pytest.mark.parametrize("N,D", [(1, 3), (31, 64), (32, 17), (33, 1), (127, 100), (129, 8),
                                 (38785, 5), (40000, 33), (98176, 5), (98177, 5), (98176, 31),
                                 (98177, 31), (163712, 5), (163713, 5), (163712, 64), (163713, 64),
                                 (163712, 32), (163713, 32)])
def test_rows(N, D, dtype):
    M = 300
    grad_check(case(M, N, D, 1, dtype), rows=np.arange(0, M, 7))


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("M,D", [(1, 3), (78, 32), (129, 64)])
@pytest.mark.parametrize("splits", [1, 2, 8, 9, 10, 16, 17, 25, 33])
def test_splits(splits, M, D, dtype):
    """Both sides of eight splits, from where the contraction loads eight of a
    row's partial sums together, with none to seven left over."""
    grad_check(case(M, 40 * 128, D, 1, dtype), split_n=splits)
