"""Images drawn band by band in shared memory, and the sizes that are drawn in global memory, against the float64
oracle renderer: one and several bands, odd widths (no 16-byte rows), one row, meshes of more triangles than the queue
holds, images too large for the bands."""
import numpy as np
import pytest

from oracle import gift_oracle as O
from synth.meshes import mesh_batch
from tests.test_gpu_render import _unstable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lat,n_lon,n_az,n_el,H,W", [
    (6, 8, 3, 1, 1, 1),       # one pixel
    (6, 8, 3, 2, 1, 64),      # one row
    (24, 48, 2, 1, 20, 21),   # 2,208 triangles through a queue of 512
    (5, 7, 1, 1, 224, 224),   # few images: many short bands
    (8, 12, 2, 1, 97, 131),   # odd width, last band shorter
    (4, 6, 1, 1, 300, 640),   # large triangles, nearly as many bands as are taken
    (4, 6, 1, 1, 640, 640),   # drawn in global memory
])
def test_bands_match_oracle(gpu_lib, n_lat, n_lon, n_az, n_el, H, W):
    V, T, vo, to = mesh_batch(1, 2, 5, 31, n_lat=n_lat, n_lon=n_lon)
    out = gpu_lib.render_views(V, T, vo, to, n_az, n_el, H, W).cpu().numpy()
    for m in range(2):
        Vm, Tm = V[vo[m]:vo[m + 1]], T[to[m]:to[m + 1]]
        ref = O.render_depth(Vm, Tm, n_az, n_el, H, W)
        ok = ~_unstable(Vm, Tm, n_az, n_el, H, W)
        assert np.array_equal(out[m][ok] < 2, ref[ok] < 2)
        assert ok.sum() == 0 or np.abs(out[m][ok] - ref[ok]).max() < 1e-4
