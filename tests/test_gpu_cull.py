"""Primitive culling of the analytic hopper and vertex pass: the masked fold
must give the full fold's bits.  The no-allocation entry point folds every
primitive; random scenes of all kinds and operations, fewer and more
primitives than a mask word holds, odd grids and an offset domain."""
import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


@pytest.mark.parametrize("n", [5, 6, 31, 32, 33, 70])
@pytest.mark.parametrize("N,lo,hi", [(47, -1.0, 1.0), (96, -0.9, 1.3)])
def test_culled_mesh_equals_full_fold(n, N, lo, hi):
    prims = synth.mixed_prims(100 + n, n - 1)
    ref = gh.Buffers(400000, keys=True)
    assert gh.polygonize_csg_noalloc(gh.csg_prims_device(prims), n, N, ref, lo=lo, hi=hi) == gh.GH_OK
    T = int(ref.counts[0])
    m = gh.polygonize(gh.CsgSdb(prims), N, lo=lo, hi=hi, keys=True)
    assert m.n_tris == T > 0
    ka, kb = ref.tri_keys[:T].cpu().numpy(), m.tri_keys.cpu().numpy()
    assert np.array_equal(meshutil.canonical_tris(ka), meshutil.canonical_tris(kb))
    ua, pa = meshutil.vertex_table(ka, ref.tri_xyz[:T].cpu().numpy())
    ub, pb = meshutil.vertex_table(kb, m.tri_xyz.cpu().numpy())
    assert np.array_equal(ua, ub) and np.array_equal(pa.view(np.uint32), pb.view(np.uint32))
    a, b = ref.stats_dict(), m.stats
    assert all(a[k] == b[k] for k in ("hop_evals", "marked_cells", "unique_vertices", "surface_cells"))
