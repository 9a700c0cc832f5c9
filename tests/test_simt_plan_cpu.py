"""Workspace of fp32 sums, worked out without a GPU: no channels need none, and
key splits never need more than 16 MiB, so that what fits the scratch of
gauss_sum_noalloc unsplit fits it split."""
import pytest

import paper_2609_04910_gb300 as gs


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2609_04910_gb300.build import build_library
    build_library()


@pytest.mark.parametrize("D", [4, 48, 128])
def test_no_channels(D):
    assert gs.gauss_sum_workspace_size(10, 10, D, 0, gs.GS_FP32) == 0


@pytest.mark.parametrize("M", [1, 33, 1000, 70001, 300000, 2000000])
@pytest.mark.parametrize("N", [1, 100, 5000, 1 << 20])
@pytest.mark.parametrize("D,C", [(3, 1), (16, 4), (32, 3), (48, 2), (64, 17), (100, 5), (128, 64)])
def test_split_sums_stay_small(M, N, D, C):
    need = gs.gauss_sum_workspace_size(M, N, D, C, gs.GS_FP32, path=gs.GS_PATH_SIMT)
    assert 0 < need <= max(16 << 20, 4 * M * C + 1023)


@pytest.mark.parametrize("N,more", [(7093, False), (7095, True), (8191, True)])
def test_one_cloud_may_need_the_tensor_cores_workspace(N, more):
    need = gs.gauss_sum_workspace_size(N, N, 3, 1, gs.GS_FP32)
    simt = gs.gauss_sum_workspace_size(N, N, 3, 1, gs.GS_FP32, path=gs.GS_PATH_SIMT)
    assert (need > simt) == more
