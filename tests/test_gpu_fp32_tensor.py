"""The FP32 evaluator's dispatch: split-BF16 products on the tensor cores up to
8 hidden layers, FP32 FMAs above.  Point lists at the edges of the 128-row
tiles (one row, one short of a tile, one more, more tiles than resident CTAs)
and the shallowest, deepest and first too deep network, against the FP64
oracle within the evaluation budget of the other point tests; and the mesh of
hopping against the mesh of enumeration (the hopper's, the vertex pass' and the
lattice's launches of the same evaluator), bit for bit."""
import numpy as np
import pytest

import meshutil
import oracle
import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


@pytest.mark.parametrize("width", [64, 128, 256])
@pytest.mark.parametrize("mid", [1, 8, 9])
def test_point_lists_at_tile_edges(width, mid):
    p = synth.pack_layers(synth.mlp_layers(3, width, mid))
    sdb = gh.MlpSdb(p, width, mid)
    o = oracle.mlp(width, mid, p.astype(np.float64))
    P = synth.uniform_points(5, 3 * 152 * 128 + 77)
    ref = o.eval_many(P[:4096].astype(np.float64))
    full = gh.eval_points(sdb, torch.from_numpy(P).cuda()).cpu().numpy()
    assert np.abs(full[:4096] - ref).max() <= parity.EVAL32
    for n in (1, 127, 128, 129, 4095):
        f = gh.eval_points(sdb, torch.from_numpy(P[:n]).cuda()).cpu().numpy()
        assert np.array_equal(f, full[:n]), n  # a row's value does not depend on its tile


@pytest.mark.parametrize("width,mid,N", [(64, 1, 40), (64, 8, 33), (128, 3, 37), (256, 8, 32), (64, 9, 33)])
def test_hopping_equals_enumeration(width, mid, N):
    p = synth.pack_layers(synth.mlp_layers(4, width, mid))
    sdb = gh.MlpSdb(p, width, mid)
    a = gh.polygonize(sdb, N, keys=True)
    b = gh.polygonize(sdb, N, keys=True, method="enum")
    ka, kb = a.tri_keys.cpu().numpy(), b.tri_keys.cpu().numpy()
    assert ka.shape[0] > 500
    assert np.array_equal(meshutil.canonical_tris(ka), meshutil.canonical_tris(kb))
    ua, pa = meshutil.vertex_table(ka, a.tri_xyz.cpu().numpy())
    ub, pb = meshutil.vertex_table(kb, b.tri_xyz.cpu().numpy())
    assert np.array_equal(ua, ub) and np.array_equal(pa.view(np.uint32), pb.view(np.uint32))
