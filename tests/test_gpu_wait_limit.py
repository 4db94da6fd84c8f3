"""What a run-out wait leaves behind: no kernel after it may read the lists it
left unfinished, whatever the scratch held before (a new SDB's uninitialised
buffers, another grid's), and every item of the launch reports it.  With the
limit at 0 every wait on the engines' own work runs out at once; nothing is
made to hang."""
import contextlib

import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


@contextlib.contextmanager
def no_waiting():
    gh.set_wait_limit_ns(0)
    try:
        yield
    finally:
        torch.cuda.synchronize()
        gh.set_wait_limit_ns(2_000_000_000)


def _tris(m):
    return meshutil.canonical_tris(m.tri_keys.cpu().numpy())


@pytest.mark.parametrize("width", [64, 128, 256])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_new_sdb_and_another_grid(width, precision):
    p = synth.mlp_params(2, width)
    eps = gh.MlpSdb(p, width).calibrate(48) if precision == "bf16" else None
    gh.release_cache()
    sdb = gh.MlpSdb(p, width)  # its scratch is allocated by the failing call
    for N in (48, 33, 70):
        with no_waiting(), pytest.raises(gh.GhError) as e:
            gh.polygonize(sdb, N, precision=precision, eps=eps, indexed=True)
        assert e.value.code == gh.GH_ERR_CUDA and "timed out" in str(e.value)
    ref = gh.MlpSdb(p, width)
    for N in (33, 70):
        m = gh.polygonize(sdb, N, precision=precision, eps=eps, indexed=True)
        r = gh.polygonize(ref, N, precision=precision, eps=eps, indexed=True)
        assert m.n_tris > 0 and np.array_equal(_tris(m), _tris(r))


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_every_item_of_a_batch_reports_it(precision):
    sdbs = [gh.MlpSdb(synth.mlp_params(s, 64), 64) for s in (1, 2, 3)] + [gh.CsgSdb(synth.csg_prims(0))]
    Ns = [40, 33, 48, 40]
    bt = gh.Batch(sdbs, Ns, [16 * n * n + 4096 for n in Ns], precision=precision, eps=1e-3, indexed=True)
    with no_waiting():
        assert bt.run(sync=False) == gh.GH_OK
        torch.cuda.synchronize()
        st = [b.stats_dict() for b in bt.bufs]
    assert [s["status"] for s in st] == [gh.GH_ERR_CUDA] * 3 + [gh.GH_OK]
    assert all(s["triangles"] == 0 for s in st[:3]) and st[3]["triangles"] > 0
    assert bt.run() == gh.GH_OK
    for b, (s, n) in enumerate(zip(sdbs, Ns)):
        single = gh.polygonize(s, n, precision=precision if b < 3 else "fp32", eps=1e-3, indexed=True)
        assert np.array_equal(_tris(bt.mesh(b)), _tris(single))


@pytest.mark.parametrize("N", [64, 200])
def test_analytic_scans(N):
    """The scans of the lists are the analytic pipeline's only waits; the
    no-allocation entry point reports them too.  The limit of 0 reaches them there
    and leaves gh_polygonize alone."""
    prims = synth.csg_prims(1)
    sdb, dev = gh.CsgSdb(prims), gh.csg_prims_device(prims)
    bufs = gh.Buffers(16 * N * N + 4096, keys=True)
    with no_waiting():
        with pytest.raises(gh.GhError) as e:
            gh.polygonize_csg_noalloc(dev, len(prims), N, bufs)
        assert e.value.code == gh.GH_ERR_CUDA and "timed out" in str(e.value)
        m = gh.polygonize(sdb, N, indexed=True)
    assert gh.polygonize_csg_noalloc(dev, len(prims), N, bufs) == gh.GH_OK
    assert np.array_equal(_tris(m), meshutil.canonical_tris(bufs.tri_keys[:int(bufs.counts[0])].cpu().numpy()))


def _surface(V):
    rng = np.random.default_rng(V)
    u = rng.standard_normal((V, 3))
    v = (0.6 * u / np.linalg.norm(u, axis=1, keepdims=True)).astype(np.float32)
    return torch.from_numpy(v).cuda(), torch.from_numpy(rng.standard_normal((V, 3)).astype(np.float32)).cuda()


@pytest.mark.parametrize("width", [64, 128, 256])
def test_calls_without_a_status_give_nan(width):
    sdb = gh.MlpSdb(synth.mlp_params(2, width), width)
    for n in (1, 129, 50001):
        P = torch.from_numpy(synth.uniform_points(3, n)).cuda()
        for precision in ("fp32", "bf16", "bf16x6"):
            ref = gh.eval_points(sdb, P, precision)
            with no_waiting():
                f = gh.eval_points(sdb, P, precision)
            assert bool(torch.isnan(f).all()), (n, precision)
            again = gh.eval_points(sdb, P, precision)
            if precision == "bf16" and width == 256:
                # its last bits depend on the tile a row falls into (the order of the
                # K-blocks follows the ring's reuse between tiles)
                assert bool(torch.isfinite(again).all())
            else:
                assert torch.equal(again, ref)
    for V in (33, 2080):
        v, dl = _surface(V)
        ref = gh.backward(sdb, v, dl)
        assert bool(torch.isfinite(ref).all())
        with no_waiting():
            g = gh.backward(sdb, v, dl)
        assert bool(torch.isnan(g).all()), V
        assert torch.equal(gh.backward(sdb, v, dl), ref)


def test_deep_networks_keep_waiting():
    p = synth.pack_layers(synth.mlp_layers(7, 64, 9))
    sdb = gh.MlpSdb(p, 64, 9)
    P = torch.from_numpy(synth.uniform_points(3, 5000)).cuda()
    v, dl = _surface(545)
    f, g = gh.eval_points(sdb, P), gh.backward(sdb, v, dl)
    with no_waiting():
        f0, g0 = gh.eval_points(sdb, P), gh.backward(sdb, v, dl)
    assert torch.equal(f0, f) and torch.equal(g0, g)


@pytest.mark.parametrize("width", [64, 256])
@pytest.mark.parametrize("n_points", [0, 4096])
def test_calibration_reports_it_and_keeps_its_bound(width, n_points):
    sdb = gh.MlpSdb(synth.mlp_params(2, width), width)
    with no_waiting(), pytest.raises(gh.GhError) as e:
        sdb.calibrate(40, n_points=n_points)
    assert e.value.code == gh.GH_ERR_CUDA and "timed out" in str(e.value)
    assert sdb.eps is None
    with pytest.raises(gh.GhError):  # no bound was stored
        gh.polygonize(sdb, 40, precision="bf16")
    assert 0.0 < sdb.calibrate(40, n_points=n_points) < 1e-2
