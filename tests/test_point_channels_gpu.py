"""Value channels and finalisation of the one-group gradient passes (quads of
coordinates, staged key rows) at the edges: widths around multiples of 4 and
up to 255, key counts around the 128-key blocks, row tiles that run unsplit
next to split ones, forward channels in quads and not, against the float64
oracle (the suite's tolerances).  (Not a single key: the suite's 2e-3 is
derived for sums in which the rounding of many operands averages out, and
the gradient of one bf16 or one uncentred fp16 key is up to 4e-3 off by the
rounding of its coordinates alone.)"""
import numpy as np
import pytest

from tests.gpu_helpers import case, forward_check, grad_check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROWS = np.concatenate([np.arange(0, 19456, 397), np.arange(19456, 20011, 13)])


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 31, 32, 33, 127, 255])
@pytest.mark.parametrize("M,N", [(70, 127), (130, 129)])
def test_gradient_widths(M, N, D, dtype):
    grad_check(case(M, N, D, 1, dtype))
    grad_check(case(M, N, D, 1, dtype), center=False)


@pytest.mark.parametrize("D", [5, 12])
def test_gradient_unsplit_and_split_rows(D):
    grad_check(case(20011, 900, D, 1, "fp16"), rows=ROWS)


@pytest.mark.parametrize("C", [5, 8, 12, 13, 64])
def test_forward_unsplit_and_split_rows(C):
    forward_check(case(20011, 900, 20, C, "bf16"), rows=ROWS)
