"""The neural adjoint at the edges of its kernels' ranges: vertex counts around
the 32-vertex stages, the 512-vertex additions and the 128-row tiles, every
width, and the shallowest, deepest and first too deep network of the tensor
path (FFMA above 8 hidden layers), against the FP64 adjoint with the tolerance
of the other adjoint tests."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


@pytest.mark.parametrize("width,mid", [(64, 1), (64, 8), (64, 9), (128, 2), (128, 8), (256, 1), (256, 5)])
@pytest.mark.parametrize("V", [1, 31, 33, 512, 545, 2080])
def test_adjoint_at_kernel_edges(width, mid, V):
    p = synth.pack_layers(synth.mlp_layers(7, width, mid))
    sdb = gh.MlpSdb(p, width, mid)
    rng = np.random.default_rng(V)
    u = rng.standard_normal((V, 3))
    verts = (u / np.linalg.norm(u, axis=1, keepdims=True) * rng.uniform(0.55, 0.65, (V, 1))).astype(np.float32)
    dl = rng.standard_normal((V, 3)).astype(np.float32)
    g = gh.backward(sdb, torch.from_numpy(verts).cuda(), torch.from_numpy(dl).cuda()).cpu().numpy().astype(np.float64)
    ref = oracle.np_adjoint(p.astype(np.float64), width, mid, verts.astype(np.float64), dl.astype(np.float64))
    scale = np.maximum(np.abs(ref), 1e-2 * np.abs(ref).max())
    assert np.isfinite(g).all()
    assert (np.abs(g - ref) <= 1e-3 * scale).all()
