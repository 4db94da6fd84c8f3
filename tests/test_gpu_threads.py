"""Several host threads polygonizing scenes of different sizes at once, each
with its own SDB and stream: no launch may depend on state another thread sets
(the culling kernel's shared-memory limit)."""
import threading

import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


def test_scenes_of_different_sizes_in_parallel():
    N, reps = 16, 3000
    scenes = [synth.mixed_prims(3, n - 1) for n in (6, 9, 12, 15, 180, 200, 230, 250)]
    sdbs = [gh.CsgSdb(p) for p in scenes]
    refs = [gh.polygonize(s, N, keys=True) for s in sdbs]
    errors = []

    def work(b):
        try:
            stream = torch.cuda.Stream()
            bufs = gh.Buffers(refs[b].n_tris + 16, keys=True)
            torch.cuda.synchronize()
            for r in range(reps):  # mostly asynchronous: the host is in the launches all the time
                assert gh.polygonize_into(sdbs[b], N, bufs, stream=stream, sync=r % 100 == 99) == gh.GH_OK
            T = int(bufs.counts[0])
            assert np.array_equal(meshutil.canonical_tris(bufs.tri_keys[:T].cpu().numpy()),
                                  meshutil.canonical_tris(refs[b].tri_keys.cpu().numpy()))
        except BaseException as e:  # noqa: BLE001 (reported by the main thread)
            errors.append((len(scenes[b]), repr(e)))

    threads = [threading.Thread(target=work, args=(b,)) for b in range(len(sdbs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
