"""The one-launch preparation of small problems gives the operands, records and
flags of the separate launches bit for bit, and keeps the problems of a batch
apart: nineteen problems fit one wave of clusters, twenty take the separate
launches, and one alone its own cluster.  Shapes whose work units (pairs of
query tiles x key tiles of all problems) number at most one per SM, so that the
fused kernel adds the same parts in the same order whatever the batch."""
import pytest

from paper_2609_04910_gb300.workloads import generate, to_device
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


def _stack(inp, name, dtype):
    return torch.stack([to_device(i[name], dtype) for i in inp]).contiguous()


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("M,N,D,C", [(512, 384, 64, 1), (500, 300, 50, 1), (257, 100, 7, 2), (512, 384, 16, 4),
                                     (100, 700, 63, 3), (1, 896, 8, 1), (300, 129, 122, 1), (200, 300, 200, 1),
                                     (60, 250, 256, 2)])
def test_sums(M, N, D, C, dtype):
    import paper_2609_04910_gb300 as gs
    inp = [generate(case(M, N, D, C, dtype, kind="offset", tau=10.0 / D), seed=s) for s in range(20)]
    q, k, v = (_stack(inp, n, dtype) for n in ("q", "k", "v"))
    tau = 10.0 / D
    separate = gs.gauss_sum_batched(q, k, v, tau)
    clusters = gs.gauss_sum_batched(q[:19].contiguous(), k[:19].contiguous(), v[:19].contiguous(), tau)
    gs.gauss_sum_device_status()
    assert not torch.equal(separate[0], separate[1])
    assert torch.equal(clusters, separate[:19])
    for b in (0, 7, 18, 19):
        assert torch.equal(gs.gauss_sum(q[b].clone(), k[b].clone(), v[b].clone(), tau), separate[b])


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("N,D", [(512, 64), (300, 20), (256, 100), (250, 64), (129, 3)])
@pytest.mark.parametrize("signs", ["halves", "mixed"])
def test_mmd2_and_one_cloud(N, D, signs, dtype):
    import paper_2609_04910_gb300 as gs
    kind = "mmd" if signs == "halves" else "normal"
    inp = [generate(case(N, N, D, 1, dtype, kind=kind, q_is_k=True), seed=s) for s in range(20)]
    x = _stack(inp, "k", dtype)
    v = _stack(inp, "v", dtype)
    w = v[..., 0].contiguous()
    separate = gs.gauss_sum_mmd2(x, w, 1.0 / D)
    assert torch.equal(gs.gauss_sum_mmd2(x[:19].contiguous(), w[:19].contiguous(), 1.0 / D), separate[:19])
    for b in (0, 11, 19):
        assert torch.equal(gs.gauss_sum_mmd2(x[b].clone(), w[b].clone(), 1.0 / D)[0], separate[b])
    if N <= 256:      # (more have eight units per problem, 160 in all)
        sums = gs.gauss_sum_batched(x, x, v, 1.0 / D)
        part = x[:19].contiguous()
        assert torch.equal(gs.gauss_sum_batched(part, part, v[:19].contiguous(), 1.0 / D), sums[:19])
    gs.gauss_sum_device_status()
