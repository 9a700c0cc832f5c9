"""Guarded fp32 sums (33 to 64 coordinates) of clustered points: close pairs
with large norms, where the exponent formed from the norms is off by units in
the last place of the norms and the SIMT kernel's differences are not.

Bound of a sum's error relative to sum |v| Phi, from float32 roundings u =
2^-24 on the tensor cores, for c q.k <= 1 and norm terms A, B <= 0.5: the norm
terms (7 additions in sequence each), their sum and the final one at most
17 u; the MMAs' partial sums, rounded towards zero, 8 full-size steps of 2 u
growing to at most 1 and the small ones: 9 u; together 26 u ln 2 < 1.1e-6;
exp2 2.4e-7; the sums of 16 keys per lane and tile, of 64 tiles and of four
column groups, with signs as they come, about sqrt(84) u = 5.5e-7 (as for the
SIMT kernel).  2e-6 in all, a fifth of the suite's fp32 tolerance."""
import math

import numpy as np
import pytest

from oracle import oracle_sum

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BOUND = 2e-6
LOG2E = 1.4426950408889634


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_04910_gb300.build import build_library
    build_library()
    torch.cuda.set_device(0)


def _clusters(M, N, D, norm, radius, seed, count=2):
    """Clusters of relative radius `radius` around +-a (or +-a, +-b, ..), with
    largest norm term (tau/2) log2(e) ||x||^2 of about `norm`."""
    rng = np.random.default_rng(seed)
    tau = 1.0 / D
    length = math.sqrt(norm / (0.5 * tau * LOG2E))
    centres = np.linalg.qr(rng.standard_normal((D, count // 2)))[0].T
    centres = np.concatenate([centres, -centres])

    def cloud(n):
        x = centres[np.arange(n) % count] * (1.0 - 2.0 * radius)
        x = x + radius * rng.standard_normal((n, D)) / math.sqrt(D)
        return (length * x).astype(np.float32)

    return cloud(M), cloud(N), tau


def _values(kind, N, rng):
    if kind == "normal":
        return rng.standard_normal((N, 1)).astype(np.float32)
    v = np.ones((N, 1), np.float32)
    if kind == "cancelling":      # within every cluster
        v[(np.arange(N) // 8) % 2 == 1] = -1.0
    return v


@pytest.mark.parametrize("kind", ["normal", "cancelling", "ones"])
@pytest.mark.parametrize("radius", [1e-4, 1e-2])
@pytest.mark.parametrize("norm", [3.9, 1.9, 1.0, 0.45])
@pytest.mark.parametrize("D", [33, 64])
def test_two_clusters(D, norm, radius, kind):
    """Just inside the norms' limit (1.9) and below it the clusters' pairs are
    close (c q.k up to 2 x norm) down to 0.5: the SIMT kernel's sums, bit for
    bit.  Below that the tensor cores', within the bound."""
    import paper_2609_04910_gb300 as gs
    M, N = 4096, 8192
    q, k, tau = _clusters(M, N, D, norm, radius, seed=11)
    v = _values(kind, N, np.random.default_rng(12))
    dq, dk, dv = (torch.from_numpy(a).cuda() for a in (q, k, v))
    got = gs.gauss_sum(dq, dk, dv, tau)
    simt = gs.gauss_sum(dq, dk, dv, tau, path=gs.GS_PATH_SIMT)
    gs.gauss_sum_device_status()
    assert torch.equal(got, simt) == (norm >= 1.0)
    rows = np.arange(0, M, 61)
    ref, den = oracle_sum(q.astype(np.float64), k.astype(np.float64), v.astype(np.float64), tau, rows=rows)
    err = np.abs(got.cpu().numpy()[rows] - ref) / den
    assert err.max() <= BOUND


@pytest.mark.parametrize("count,simt", [(16, True), (64, True)])
def test_many_clusters(count, simt):
    """One pair in `count` is close: more than one in 256."""
    import paper_2609_04910_gb300 as gs
    q, k, tau = _clusters(4096, 8192, 64, 1.5, 1e-2, seed=13, count=count)
    v = _values("normal", 8192, np.random.default_rng(14))
    dq, dk, dv = (torch.from_numpy(a).cuda() for a in (q, k, v))
    same = torch.equal(gs.gauss_sum(dq, dk, dv, tau),
                       gs.gauss_sum(dq, dk, dv, tau, path=gs.GS_PATH_SIMT))
    assert same == simt


@pytest.mark.parametrize("M,N,D,C", [(4096, 4300, 33, 1), (16384, 16384, 64, 1), (9000, 3000, 40, 3)])
def test_normal_points_stay_on_the_tensor_cores(M, N, D, C):
    import paper_2609_04910_gb300 as gs
    gen = torch.Generator(device="cuda").manual_seed(15)
    q, k, v = (torch.randn(*s, generator=gen, device="cuda") for s in ((M, D), (N, D), (N, C)))
    got = gs.gauss_sum(q, k, v, 1.0 / D)
    assert not torch.equal(got, gs.gauss_sum(q, k, v, 1.0 / D, path=gs.GS_PATH_SIMT))
