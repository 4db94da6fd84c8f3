"""FP32 networks whose layers are not dense: identities, selections, pruned
rows.  The split-BF16 engine adds back what its truncated accumulator loses on
average, by the number of terms an output has; where a layer's sums are exact
(powers of two selecting one input each) it must add nothing, so f has the bits of
exact arithmetic, and with few terms the mean error must stay near zero."""
import numpy as np
import pytest

import meshutil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402

BARE = dict(r0=0.0, alpha=1.0, beta=1.0, radial=False)


def _selections(width, mid, seed):
    """W0 with one coordinate per unit, hidden layers a permutation times powers
    of two, the output one unit: every f is one product and exact scalings."""
    rng = np.random.default_rng(seed)
    W0 = np.zeros((width, 3))
    W0[np.arange(width), np.arange(width) % 3] = rng.uniform(0.5, 1.5, width) * rng.choice([-1, 1], width)
    layers = [(W0, np.zeros(width))]
    for _ in range(mid):
        M = np.zeros((width, width))
        M[np.arange(width), rng.permutation(width)] = 2.0 ** rng.integers(-2, 3, width)
        layers.append((M, np.zeros(width)))
    wo = np.zeros((1, width))
    wo[0, int(rng.integers(width))] = 1.0
    layers.append((wo, np.zeros(1)))
    return synth.pack_layers(layers).astype(np.float32)


def _exact_f32(p, width, mid, P):
    """f of such a network: layer 0 rounded once to float32, the rest exact."""
    layers = synth.unpack_layers(p, width, mid)
    x = np.maximum((P.astype(np.float64) @ layers[0][0].T.astype(np.float64)).astype(np.float32), 0).astype(np.float64)
    for M, _ in layers[1:-1]:
        x = np.maximum(x @ M.T.astype(np.float64), 0)
    return (x @ layers[-1][0].T.astype(np.float64))[:, 0]


@pytest.mark.parametrize("width", [64, 128, 256])
@pytest.mark.parametrize("mid", [1, 5, 8])
def test_exact_layers_stay_exact(width, mid):
    P = synth.uniform_points(9, 4096)
    t = torch.from_numpy(P).cuda()
    for seed in range(3):
        p = _selections(width, mid, seed)
        ref = _exact_f32(p, width, mid, P)
        assert (ref > 0).mean() > 0.2
        for precision in ("fp32", "bf16x6"):
            f = gh.eval_points(gh.MlpSdb(p, width, mid, **BARE), t, precision).cpu().numpy().astype(np.float64)
            assert np.array_equal(f, ref), (seed, precision)


@pytest.mark.parametrize("width", [64, 128, 256])
@pytest.mark.parametrize("kind,terms", [("any", 1), ("any", 2), ("any", 8), ("any", 32), ("pow2", 2), ("pow2", 8),
                                        ("pow2", 32)])
def test_few_terms_have_no_mean_error(width, kind, terms):
    """One hidden layer, one output with `terms` positive weights and a bias: the
    mean error over 256 such layers, in units of the result's last place.  The
    truncation is 0 to 0.65 units on average and corrected within 0.07 of it where
    it was measured (positive weights, half of the activations zero).  The
    correction, mostly below half a unit, comes with the bias in one rounding,
    which is the same for all points of a layer whose results share an exponent:
    a uniform error of deviation 0.29 per layer, 0.018 over 256, three of which
    and the 0.07 are within the bound."""
    errs = []
    for seed in range(256):
        rng = np.random.default_rng(100 * seed + terms)
        W0 = np.zeros((width, 3))
        W0[np.arange(width), np.arange(width) % 3] = rng.standard_normal(width)
        M = np.zeros((width, width))
        at = rng.choice(width, terms, replace=False)
        M[0, at] = 2.0 ** rng.integers(-4, 3, terms) if kind == "pow2" else np.abs(rng.standard_normal(terms)) + 0.1
        wo = np.zeros((1, width))
        wo[0, 0] = 1.0
        bias = np.zeros(width)
        bias[0] = rng.uniform(0.01, 0.02)
        p = synth.pack_layers([(W0, np.zeros(width)), (M, bias), (wo, np.zeros(1))]).astype(np.float32)
        P = synth.uniform_points(seed, 256)
        f = gh.eval_points(gh.MlpSdb(p, width, 1, **BARE), torch.from_numpy(P).cuda()).cpu().numpy().astype(np.float64)
        l = synth.unpack_layers(p, width, 1)
        x = np.maximum((P.astype(np.float64) @ l[0][0].T.astype(np.float64)).astype(np.float32), 0).astype(np.float64)
        acc = x @ l[1][0][0].astype(np.float64)
        ref = acc + float(l[1][1][0])
        on = acc > 0
        errs.append((f[on] - ref[on]) / 2.0 ** (np.floor(np.log2(ref[on])) - 23))
    e = np.concatenate(errs)
    print("width %d, %d %s terms: mean %.3f, deviation %.3f units" % (width, terms, kind, e.mean(), e.std()))
    assert abs(e.mean()) < 0.15


@pytest.mark.parametrize("width", [64, 128, 256])
def test_adjoint_through_exact_layers(width):
    """s_v of one vertex through five selecting layers: the delta chain is exact,
    so dL/db_out = -(dL/dv . g) / |g|^2 has the roundings of that formula only
    (g exact; at most about eight of 2^-24 each)."""
    p = _selections(width, 5, 1)
    sdb = gh.MlpSdb(p, width, 5, **BARE)
    layers = [w for w, _ in synth.unpack_layers(p, width, 5)]
    rng = np.random.default_rng(0)
    seen = 0
    for _ in range(64):
        v = rng.uniform(-1, 1, (1, 3)).astype(np.float32)
        d = rng.standard_normal((1, 3)).astype(np.float32)
        zs, x = [], v.astype(np.float64)
        for M in layers[:-1]:
            z = x @ M.T.astype(np.float64)
            zs.append(z)
            x = np.maximum(z, 0)
        g = layers[-1].astype(np.float64)
        for M, z in zip(reversed(layers[:-1]), reversed(zs)):
            g = (g * (z > 0)) @ M.astype(np.float64)
        if not (g * g).sum() > 0:
            continue
        seen += 1
        ref = -(d.astype(np.float64) * g).sum() / (g * g).sum()
        out = gh.backward(sdb, torch.from_numpy(v).cuda(), torch.from_numpy(d).cuda()).cpu().numpy()
        assert abs(float(out[-1]) - ref) <= 8 * 2.0 ** -24 * abs(ref)
    assert seen >= 10


@pytest.mark.parametrize("width,mid,N", [(64, 8, 33), (128, 3, 37), (256, 5, 40)])
def test_pruned_network_same_mesh_in_every_launch(width, mid, N):
    """Pruned hidden layers (a tenth of the weights left, some rows empty, one
    layer dense): hopping, vertex values, refinement, enumeration and a batch with
    a dense network are launches of one evaluator and give one mesh."""
    rng = np.random.default_rng(width)
    layers = synth.mlp_layers(4, width, mid)
    for l in range(1, mid + 1):
        if l != 2:
            M = layers[l][0] * (rng.random((width, width)) < 0.1)
            layers[l] = (M / np.linalg.norm(M, 2), layers[l][1])
    p = synth.pack_layers(layers)
    sdb = gh.MlpSdb(p, width, mid)
    dense = gh.MlpSdb(synth.pack_layers(synth.mlp_layers(5, width, mid)), width, mid)
    eps = sdb.calibrate(N) if mid <= (7 if width == 256 else 8) else None
    ref = gh.polygonize(sdb, N, keys=True)
    assert ref.n_tris > 500
    bt = gh.Batch([dense, sdb], [N + 3, N], [20 * N * N + 4096] * 2, keys=True)
    assert bt.run() == gh.GH_OK
    meshes = [gh.polygonize(sdb, N, keys=True, method="enum"), bt.mesh(1)]
    if eps is not None:
        meshes.append(gh.polygonize(sdb, N, keys=True, precision="bf16x6", eps=eps))
    ka = ref.tri_keys.cpu().numpy()
    ua, pa = meshutil.vertex_table(ka, ref.tri_xyz.cpu().numpy())
    for m in meshes:
        kb = m.tri_keys.cpu().numpy()
        assert np.array_equal(meshutil.canonical_tris(ka), meshutil.canonical_tris(kb))
        ub, pb = meshutil.vertex_table(kb, m.tri_xyz.cpu().numpy())
        assert np.array_equal(ua, ub) and np.array_equal(pa.view(np.uint32), pb.view(np.uint32))
