"""What a mesh keeps on the device: the first guess of its triangle buffer."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2111_05778_gb300 import gh, synth  # noqa: E402


def test_first_guess_of_the_triangle_buffer():
    N = 96
    for sdb, per_column in ((gh.CsgSdb(synth.sphere_prims(0.5)), 4), (gh.CsgSdb(synth.csg_prims(0)), 8),
                            (gh.MlpSdb(synth.mlp_params(1, 64), 64), 4)):
        m = gh.polygonize(sdb, N)
        assert 0 < m.n_tris <= per_column * N * N
        assert m.tri_xyz.untyped_storage().nbytes() == 36 * (per_column * N * N + 4096)
