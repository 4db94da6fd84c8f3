"""Primitives much larger than the domain (a ground sphere, walls): their
distances round by far more than the domain's coordinates do, and the culling
masks must still give the full fold's bits.  Two spheres of radius ~2e4 touch at
the corner of a block of cells, where the two distances are furthest from their
values at the block's centre; the no-allocation entry point folds everything."""
import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


def _touching(seed, N, radius):
    rng = np.random.default_rng(seed)
    edge, n3 = (N + 31) // 32, np.ones(3) / np.sqrt(3.0)
    p = -1.0 + 2.0 / N * edge * float(rng.integers(8, 24)) * np.ones(3)
    rows = []
    for sgn in (-1, 1):
        r = float(np.float32(radius * rng.uniform(0.5, 1.5)))
        rows.append(synth.sphere_prims(r, p + sgn * n3 * r)[0])
    rows += [synth.sphere_prims(0.5, rng.uniform(6, 9, 3))[0] for _ in range(4)]
    return np.array(rows)


@pytest.mark.parametrize("N,seed,radius", [(N, s, r) for N in (32, 64) for s in (0, 2, 3, 4) for r in (20.0, 2e4)] +
                         [(256, 23, 2e5)])
def test_large_spheres_keep_the_full_folds_bits(N, seed, radius):
    prims = _touching(seed, N, radius)
    ref = gh.Buffers(1000000, keys=True)
    assert gh.polygonize_csg_noalloc(gh.csg_prims_device(prims), len(prims), N, ref) == gh.GH_OK
    T = int(ref.counts[0])
    m = gh.polygonize(gh.CsgSdb(prims), N, keys=True)
    a, b = ref.stats_dict(), m.stats
    assert all(a[k] == b[k] for k in ("hop_evals", "marked_cells", "unique_vertices", "surface_cells", "triangles"))
    if T == 0:  # (the rounding of such radii can close the gap between the spheres)
        return
    ka, kb = ref.tri_keys[:T].cpu().numpy(), m.tri_keys.cpu().numpy()
    assert np.array_equal(meshutil.canonical_tris(ka), meshutil.canonical_tris(kb))
    ua, pa = meshutil.vertex_table(ka, ref.tri_xyz[:T].cpu().numpy())
    ub, pb = meshutil.vertex_table(kb, m.tri_xyz.cpu().numpy())
    assert np.array_equal(ua, ub) and np.array_equal(pa.view(np.uint32), pb.view(np.uint32))
