"""FMA kernel with the query rows in tensor memory (rows too wide for the
augmented layout): one S tile per query tile, each handed over by itself.
Few key tiles (fewer than the pipeline's stages, and just as many), several
segments per block, one to four channels in quad records, two and three
stages, against the float64 oracle and bit for bit on repeats."""
import numpy as np
import pytest

from tests.gpu_helpers import case, forward_check, to_device  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("C", [1, 2, 3, 4])
@pytest.mark.parametrize("D,dtype", [(128, "fp16"), (150, "bf16"), (256, "fp16")])
@pytest.mark.parametrize("M,N,split_n", [(5, 1, 0), (257, 129, 1), (130, 384, 1), (600, 1000, 3),
                                         (256, 2000, 1)])
def test_few_key_tiles_and_segments(M, N, split_n, D, dtype, C):
    forward_check(case(M, N, D, C, dtype), split_n=split_n)


@pytest.mark.parametrize("D,C", [(128, 1), (256, 4), (200, 2)])
def test_many_units_repeat_bitwise(D, C):
    import paper_2609_04910_gb300 as gs
    gen = torch.Generator(device="cuda").manual_seed(D + C)
    q = (0.1 * torch.randn(12000, D, generator=gen, device="cuda")).half()
    k = (0.1 * torch.randn(20000, D, generator=gen, device="cuda")).half()
    v = torch.randn(20000, C, generator=gen, device="cuda").half()
    first = gs.gauss_sum(q, k, v, 10.0 / D)
    for _ in range(6):
        again = gs.gauss_sum(q, k, v, 10.0 / D)
        assert torch.equal(first, again)
    gs.gauss_sum_device_status()
    rows = np.arange(0, 12000, 499)
    qd, kd, vd = (t.double() for t in (q[rows], k, v))
    d2 = torch.cdist(qd, kd) ** 2
    phi = torch.exp(-5.0 / D * d2)
    err = (first[rows].double() - phi @ vd).abs() / (phi @ vd.abs())
    assert err.max().item() <= 2e-3
