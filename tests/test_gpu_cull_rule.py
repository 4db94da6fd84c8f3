"""Where the culling masks are built: not for unions of few spheres or on small
grids, whose tight loop the masks slow down, nor for scenes with a primitive
without a bounding radius; and the mesh does not depend on it, also when one SDB
changes sides with N, when its scratch comes from the pool, and in a batch of
scenes of both kinds."""
import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


def _spheres(n, seed=0):
    rng = np.random.default_rng(seed)
    return np.concatenate([synth.sphere_prims(rng.uniform(0.05, 0.3), rng.uniform(-0.6, 0.6, 3)) for _ in range(n)])


def _skewed():
    prims = synth.mixed_prims(5, 11).copy()
    prims[3, 8] += 3e-5  # accepted as a rotation, but too far from one for a bounding radius
    return prims


SCENES = {"spheres 24": lambda: _spheres(24), "spheres 128": lambda: _spheres(128), "mixed 12": lambda: synth.mixed_prims(5, 11),
          "skewed 12": _skewed, "spheres 64 and 5": lambda: np.concatenate([_spheres(64), synth.primitive_scene(1)[1:6]])}
MASKS = {"spheres 24": (False, False), "spheres 128": (False, True), "mixed 12": (True, True), "skewed 12": (False, False),
         "spheres 64 and 5": (False, True)}
NS = (48, 160)


def _tris(keys):
    return meshutil.canonical_tris(keys.cpu().numpy())


@pytest.mark.parametrize("name", list(SCENES))
def test_masks_where_they_pay_and_one_mesh(name):
    prims = SCENES[name]()
    plain = gh.CsgSdb(_spheres(3))
    gh.polygonize(plain, 48)
    base = gh.last_profile()[0]
    sdb = gh.CsgSdb(prims)
    for N, masks in list(zip(NS, MASKS[name])) + [(NS[0], MASKS[name][0])]:
        ref = gh.Buffers(24 * N * N + 4096, keys=True)
        assert gh.polygonize_csg_noalloc(gh.csg_prims_device(prims), len(prims), N, ref) == gh.GH_OK
        T = int(ref.counts[0])
        m = gh.polygonize(sdb, N, keys=True)
        assert gh.last_profile()[0] == base + (1 if masks else 0), (N, masks)
        assert m.n_tris == T > 0 and np.array_equal(_tris(m.tri_keys), _tris(ref.tri_keys[:T]))
        assert m.stats["hop_evals"] == ref.stats_dict()["hop_evals"]


def test_batch_of_both_kinds_with_pooled_scratch():
    gh.release_cache()
    scenes = [f() for f in SCENES.values()]
    for _ in range(2):  # the second time the scratch, masks included, comes from the pool
        sdbs = [gh.CsgSdb(p) for p in scenes]
        for Ns in ([NS[0]] * len(scenes), [NS[1]] * len(scenes), [48, 160, 48, 160, 48]):
            bt = gh.Batch(sdbs, Ns, [24 * n * n + 4096 for n in Ns], keys=True)
            assert bt.run() == gh.GH_OK
            for b, (p, n) in enumerate(zip(scenes, Ns)):
                ref = gh.Buffers(24 * n * n + 4096, keys=True)
                assert gh.polygonize_csg_noalloc(gh.csg_prims_device(p), len(p), n, ref) == gh.GH_OK
                assert np.array_equal(_tris(bt.mesh(b).tri_keys), _tris(ref.tri_keys[:int(ref.counts[0])])), (b, n)
        for s in sdbs:
            s.close()
