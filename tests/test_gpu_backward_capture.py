"""gh_backward under CUDA-graph capture: after one call of an SDB no later one
allocates, whatever its number of vertices, so it can be captured; and the
work buffer a captured call holds is not moved by larger calls nor by the
scratch the SDB takes from the pool for a polygonization."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


def _surface(V, seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((V, 3))
    v = (0.6 * u / np.linalg.norm(u, axis=1, keepdims=True)).astype(np.float32)
    return torch.from_numpy(v).cuda(), torch.from_numpy(rng.standard_normal((V, 3)).astype(np.float32)).cuda()


@pytest.mark.parametrize("width,mid", [(64, 5), (128, 2), (64, 9)])
def test_captured_backward_survives_other_calls(width, mid):
    gh.release_cache()
    # a pooled scratch with an adjoint buffer of its own, larger than this SDB's
    other = gh.MlpSdb(synth.mlp_params(1, 256), 256)
    gh.polygonize(other, 40)
    gh.backward(other, *_surface(100, 0))
    p = synth.pack_layers(synth.mlp_layers(7, width, mid))
    sdb = gh.MlpSdb(p, width, mid)
    gh.backward(sdb, *_surface(100, 1))  # warm-up, fewer vertices than the captured call
    v, dl = _surface(9000, 2)
    ref = gh.backward(sdb, v, dl)
    del sdb
    sdb = gh.MlpSdb(p, width, mid)
    gh.backward(sdb, *_surface(100, 1))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g = gh.backward(sdb, v, dl)
    other.close()
    gh.backward(sdb, *_surface(60000, 3))
    gh.polygonize(sdb, 40)
    fill = torch.full((1 << 24,), 7.0, device="cuda")
    g.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(g, ref) and bool((fill == 7.0).all())
