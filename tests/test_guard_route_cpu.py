"""Which fp32 sums of 33 to 64 coordinates launch both paths, seen from the
workspace they ask for: not those of few queries or few keys, where writing
the tensor cores' operands costs more than the SIMT kernel's whole sum, nor
those too small to repay the launches."""
import pytest

import paper_2609_04910_gb300 as gs


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2609_04910_gb300.build import build_library
    build_library()


def _guarded(M, N, D, C):
    both = gs.gauss_sum_workspace_size(M, N, D, C, gs.GS_FP32)
    simt = gs.gauss_sum_workspace_size(M, N, D, C, gs.GS_FP32, path=gs.GS_PATH_SIMT)
    # Operands of both arrays: hi and lo halves of 64 coordinates per point.
    assert both == simt or both > simt + 512 * (M + N)
    return both != simt


@pytest.mark.parametrize("D", [33, 48, 50, 64])
@pytest.mark.parametrize("M,N", [(1 << 20, 32), (32, 1 << 20), (1 << 18, 64), (64, 1 << 18),
                                 (128, 1 << 17), (4095, 4096), (1000, 1000)])
def test_simt_alone(M, N, D):
    assert not _guarded(M, N, D, 1)


@pytest.mark.parametrize("D,C", [(33, 1), (48, 4), (50, 1), (64, 2)])
@pytest.mark.parametrize("M,N", [(16384, 16384), (3000, 60001), (60000, 2000), (100000, 100000)])
def test_guarded(M, N, D, C):
    assert _guarded(M, N, D, C)


def test_other_widths_and_channels():
    assert not _guarded(20000, 20000, 65, 1)
    assert not _guarded(20000, 20000, 64, 5)
