"""fp32 SIMT forward kernel against the float64 oracle at the edges of its
register tiles (4, 8, 16, 24, 32, 48, 64 or 128 coordinates, shared by one,
two or four lanes), of its row blocks (512 to 64 rows), key tiles and
channel blocks (1, 2 or 4), and on both sides of the size from which forward
sums of few coordinates go to the tensor cores.  Tolerance: the suite's fp32
bound."""
import numpy as np
import pytest

from tests.gpu_helpers import case, forward_check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("D", [1, 3, 4, 5, 8, 9, 17, 24, 25, 31, 33, 48, 49, 63, 65, 96, 127])
@pytest.mark.parametrize("M,N,C", [(513, 321, 1), (257, 63, 2), (129, 1000, 3), (1, 5, 6),
                                   (1100, 700, 1), (63, 2000, 4)])
def test_register_tiles_and_channel_blocks(D, M, N, C):
    forward_check(case(M, N, D, C, "fp32"))


@pytest.mark.parametrize("D,split_n", [(16, 3), (50, 40), (128, 7)])
def test_forced_key_splits(D, split_n):
    forward_check(case(300, 2500, D, 1, "fp32"), split_n=split_n)


@pytest.mark.parametrize("D,pairs", [(4, 1 << 26), (5, 1 << 25), (8, 1 << 25), (9, 1 << 25)])
def test_size_switch_to_the_tensor_cores(D, pairs):
    rows = np.arange(0, 4096, 37)
    for N in (pairs // 4096 - 1, pairs // 4096):
        forward_check(case(4096, N, D, 1, "fp32"), rows=rows)
