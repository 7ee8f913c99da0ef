"""Directions with components whose reciprocal is not a finite number (subnormal ones): a ray goes where the ray with a
component of 1e-20 goes, to the last bit, in every form that steps over cells."""
import numpy as np
import pytest

import scenegen as sg
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _scene(tiny):
    rng = np.random.default_rng(5)
    conc = rng.uniform(0.0, 4.0, (1, 16, 16, 16)).astype(np.float32)
    conc[0, 4:8] = 0.0   # empty cells to leap over
    conc[0, 12:14, :, 8:] = 0.0
    sc = sg.cfg1_homogeneous_cube(n_paths=20_000, film=8)
    sc["medium"] = sg.grid_medium(conc, sigma_s=0.0)
    # on a plane between voxels and between cells; the film looks down the same way
    sc["sources"] = [sg.pencil_beam((0.5, 0.5, 1.0), (tiny, 0.0, -1.0), [490.0])]
    sc["sensor"] = sg.ortho_sensor(8, 8, (0, 0, 1), (1, 0, 0), (0, 1, 0), (tiny, 0, 1))
    return sc


@pytest.mark.parametrize("tiny", [5e-39, 1e-40, 1.4e-45, 2e-38, -5e-39, -1e-40])
@pytest.mark.parametrize("kw", [{}, {"macro_cell": 4}, {"macro_cell": 1}, {"skip_cell": 1}, {"skip_cell": 4}])
def test_a_subnormal_component_is_a_small_one(tiny, kw):
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    out = []
    for t in (tiny, np.copysign(1e-20, tiny)):
        S = Scene(_scene(float(t)))
        for form in ("plain", "wavefront", "wavefront_warp"):
            film = S.render(form=form, **kw).cpu().numpy().copy()
            out.append((film, S.read()))
        S.close()
    assert out[0][1]["absorbed"].sum() > 0.1
    for (f, r), (f0, r0) in zip(out[:3], out[3:]):
        assert r["counters"] == r0["counters"]
        assert all(np.array_equal(r[k], r0[k]) for k in ("face", "absorbed", "emitted"))
        assert np.array_equal(f, f0)
