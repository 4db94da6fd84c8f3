"""A captured batch graph stays valid while its SDBs are used otherwise: a later
call on one of them that needs no larger scratch must not move a buffer the
graph holds.  The analytic scene's culling masks have more blocks on some
smaller grids (N = 40: 20 per axis, N = 32: 32; N = 200: 29, N = 64: 32)."""
import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


@pytest.mark.parametrize("N,smaller", [(40, 32), (200, 64)])
@pytest.mark.parametrize("n_prims", [6, 36, 70])
def test_graph_replay_after_a_smaller_call(N, smaller, n_prims):
    gh.release_cache()  # a pooled buffer could be large enough
    prims = synth.csg_prims(1) if n_prims == 36 else synth.mixed_prims(3, n_prims - 1)
    sdb = gh.CsgSdb(prims)
    ref = gh.polygonize(gh.CsgSdb(prims), N, keys=True)
    gh.release_cache()
    bt = gh.Batch([sdb], [N], [16 * N * N + 4096], keys=True)
    bt.capture()
    small = gh.polygonize(sdb, smaller, keys=True)
    assert small.n_tris > 0
    # whatever the smaller call gave back would be handed out again here
    fill = [torch.full((1 << 18,), 0x5A5A5A5A, dtype=torch.int32, device="cuda") for _ in range(8)]
    bt.bufs[0].counts.zero_()
    bt.replay()
    torch.cuda.synchronize()
    m = bt.mesh(0)
    assert np.array_equal(meshutil.canonical_tris(m.tri_keys.cpu().numpy()),
                          meshutil.canonical_tris(ref.tri_keys.cpu().numpy()))
    assert all(bool((f == 0x5A5A5A5A).all()) for f in fill)
