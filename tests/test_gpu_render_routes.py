"""Depth views drawn band by band and in global memory are the same bits: one mesh alone (few images of many triangles:
global memory), the same mesh in a large batch (bands), small and large triangles mixed."""
import numpy as np
import pytest

from synth.meshes import mesh_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lat,n_lon,H,W", [(60, 80, 224, 224), (60, 80, 97, 131), (40, 60, 33, 20)])
@pytest.mark.parametrize("extra", [0, 3])
def test_alone_and_in_a_batch(gpu_lib, n_lat, n_lon, H, W, extra):
    V, T, vo, to = mesh_batch(3, 1, 5, 31, n_lat=n_lat, n_lon=n_lon)
    g = np.random.default_rng(5)
    V = np.concatenate([V, g.uniform(-1, 1, (3 * extra, 3)).astype(V.dtype)])  # large triangles through the surface
    T = np.concatenate([T, (len(V) - 3 * extra + np.arange(3 * extra).reshape(-1, 3)).astype(T.dtype)])
    one = gpu_lib.render_views(V, T, [0, len(V)], [0, len(T)], 2, 1, H, W).cpu().numpy()
    M = 128
    many = gpu_lib.render_views(np.tile(V, (M, 1)), np.tile(T, (M, 1)), np.arange(M + 1) * len(V),
                                np.arange(M + 1) * len(T), 2, 1, H, W).cpu().numpy()
    assert (one < 2).any()
    for m in (0, 77, M - 1):
        assert np.array_equal(many[m], one[0])
