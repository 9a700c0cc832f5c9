"""What the Python entry points refuse before they reach the C ABI."""
import pytest

import paper_2609_04910_gb300 as gs

torch = pytest.importorskip("torch")


class _OnDevice(torch.Tensor):
    """A host tensor that passes for a CUDA tensor; a call that gets past the
    checks would fail on its pointers' first use, so none may."""

    is_cuda = True


@pytest.mark.parametrize("dtype", [torch.float64, torch.float16, torch.bfloat16, torch.int32])
def test_vjp_upstream_of_another_type_is_a_value_error(dtype):
    q, k, v, g = (torch.zeros(4, n, dtype=t).as_subclass(_OnDevice)
                  for n, t in ((2, torch.float16), (2, torch.float16), (1, torch.float16),
                               (1, dtype)))
    with pytest.raises(ValueError, match="g must be float32"):
        gs.gauss_sum_vjp(q, k, v, g, 1.0)
