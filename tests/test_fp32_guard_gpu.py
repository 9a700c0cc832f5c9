"""Large fp32 sums of 33 to 64 coordinates: the guarded pair of paths (3xTF32
MMAs with the query rows in tensor memory, or the SIMT kernel) on both sides
of the guard and of the size switch, against the float64 oracle with the
suite's fp32 tolerance; and what stays on the SIMT path."""
import numpy as np
import pytest

from oracle import oracle_sum
from paper_2609_04910_gb300.workloads import device_inputs, generate
from tests.gpu_helpers import TOL, case, forward_check, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROWS = np.arange(0, 4096, 41)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("D,C", [(33, 1), (40, 2), (63, 3), (64, 4), (64, 1), (65, 1)])
@pytest.mark.parametrize("M,N", [(4096, 4097), (4100, 4223), (300, 60001)])
def test_guarded_parity(D, C, M, N):
    forward_check(case(M, N, D, C, "fp32"), rows=ROWS[ROWS < M])


@pytest.mark.parametrize("D", [33, 64])
def test_size_switch(D):
    for N in (4095, 4096):
        forward_check(case(4096, N, D, 1, "fp32"), rows=ROWS)


def test_aliased_and_offset_clouds():
    forward_check(case(5000, 5000, 48, 1, "fp32", kind="mmd", q_is_k=True), rows=ROWS)
    forward_check(case(4096, 5000, 64, 2, "fp32", kind="offset", tau=10.0 / 64), rows=ROWS)


@pytest.mark.parametrize("center", [True, False])
def test_guard_leaves_large_norms_to_the_simt_kernel(center):
    """tau = 1: (c/2)||x||^2 is about 46, beyond the guard's 4; an
    uncentred common offset likewise.  The result is then the SIMT kernel's
    own, bit for bit; within the guard it differs from it by rounding."""
    import paper_2609_04910_gb300 as gs
    inp = generate(case(4096, 4500, 64, 1, "fp32"), seed=3)
    q, k, v = device_inputs(inp)
    simt = gs.gauss_sum(q, k, v, 1.0, path=gs.GS_PATH_SIMT)
    assert torch.equal(gs.gauss_sum(q, k, v, 1.0, center=center), simt)
    simt = gs.gauss_sum(q, k, v, 1.0 / 64, path=gs.GS_PATH_SIMT)
    near = gs.gauss_sum(q, k, v, 1.0 / 64, center=center)
    assert not torch.equal(near, simt)
    ref, den = oracle_sum(inp["q64"], inp["k64"], inp["v64"], 1.0 / 64, rows=ROWS)
    assert rel_err(near.cpu().numpy()[ROWS], ref, den) <= TOL["fp32"]
    qs, ks = q + 8.0, k + 8.0
    shifted = gs.gauss_sum(qs, ks, v, 1.0 / 64, center=center)
    same = torch.equal(shifted, gs.gauss_sum(qs, ks, v, 1.0 / 64, path=gs.GS_PATH_SIMT))
    assert same == (not center)


def test_not_a_number_takes_the_simt_path():
    import paper_2609_04910_gb300 as gs
    inp = generate(case(4096, 4500, 40, 1, "fp32"), seed=4)
    q, k, v = device_inputs(inp)
    q[17, 3] = float("nan")
    got = gs.gauss_sum(q, k, v, 1.0 / 40)
    want = gs.gauss_sum(q, k, v, 1.0 / 40, path=gs.GS_PATH_SIMT)
    assert torch.isnan(got[17]).all() and torch.isnan(got).sum() == 1
    assert torch.equal(torch.nan_to_num(got), torch.nan_to_num(want))


def test_scratch_limits_keep_the_simt_path():
    """A caller's workspace or the no-allocation scratch too small for the
    guarded pair runs the SIMT path as before."""
    import paper_2609_04910_gb300 as gs
    inp = generate(case(33000, 40000, 64, 1, "fp32"), seed=5)
    q, k, v = device_inputs(inp)
    simt = gs.gauss_sum(q, k, v, 1.0 / 64, path=gs.GS_PATH_SIMT)
    need = gs.gauss_sum_workspace_size(33000, 40000, 64, 1, gs.GS_FP32)
    assert need > 32 * 1024 * 1024
    assert torch.equal(gs.gauss_sum_noalloc(q, k, v, 1.0 / 64), simt)
    small = torch.empty(gs.gauss_sum_workspace_size(33000, 40000, 64, 1, gs.GS_FP32,
                                                    path=gs.GS_PATH_SIMT),
                        dtype=torch.uint8, device="cuda")
    assert torch.equal(gs.gauss_sum(q, k, v, 1.0 / 64, workspace=small), simt)
    full = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert torch.equal(gs.gauss_sum(q, k, v, 1.0 / 64, workspace=full),
                       gs.gauss_sum(q, k, v, 1.0 / 64))


@pytest.mark.parametrize("M,N,D,C", [(16384, 16384, 64, 1), (16384, 16384, 33, 4),
                                     (5000, 30001, 48, 2)])
def test_many_key_tiles_repeat_bitwise(M, N, D, C):
    """Long sequences of tf32 MMAs with the S tiles handed back as soon as they
    are in registers: repeated calls agree bit for bit."""
    import paper_2609_04910_gb300 as gs
    q, k, v = device_inputs(generate(case(M, N, D, C, "fp32"), seed=6))
    first = gs.gauss_sum(q, k, v, 1.0 / D)
    again = [gs.gauss_sum(q, k, v, 1.0 / D) for _ in range(20)]
    gs.gauss_sum_device_status()
    assert all(torch.equal(first, a) for a in again)
