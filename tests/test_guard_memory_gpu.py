"""Guarded fp32 sums whose workspace for both paths cannot be allocated: the
SIMT kernel alone, as before there was a second path; and no workspace at all
is out of memory."""
import pytest

from paper_2609_04910_gb300.workloads import device_inputs, generate
from tests.gpu_helpers import case

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


def test_guarded_sum_without_room_for_both_paths():
    import paper_2609_04910_gb300 as gs
    from paper_2609_04910_gb300._binding import testing_fail_next_allocations
    q, k, v = device_inputs(generate(case(4200, 4500, 48, 2, "fp32"), seed=21))
    simt = gs.gauss_sum(q, k, v, 1.0 / 48, path=gs.GS_PATH_SIMT)
    both = gs.gauss_sum(q, k, v, 1.0 / 48)
    assert not torch.equal(both, simt)
    try:
        testing_fail_next_allocations(1)
        assert torch.equal(gs.gauss_sum(q, k, v, 1.0 / 48), simt)
        assert torch.equal(gs.gauss_sum(q, k, v, 1.0 / 48), both)
        testing_fail_next_allocations(2)
        with pytest.raises(gs.GaussSumError) as ei:
            gs.gauss_sum(q, k, v, 1.0 / 48)
        assert ei.value.status == 3                # GS_ERR_OUT_OF_MEMORY
    finally:
        testing_fail_next_allocations(0)
