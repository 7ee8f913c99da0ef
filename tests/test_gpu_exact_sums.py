"""Counters carried out of 32-bit words against a form that counts in 64 bits, and maxima over grids that hold
negative zeros."""
import numpy as np
import pytest
import torch

import scenegen as sg
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
FORMS = ("plain", "wavefront", "wavefront_warp", "wavefront_pool")


@pytest.mark.parametrize("n_paths,max_events", [(33, 40_000), (700, 20_000)])
def test_carried_counters_against_a_form_that_counts_in_64_bits(n_paths, max_events):
    """One wavelength a path of the plain hero form: its counters are 64-bit words throughout."""
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    sc = sg.cfg1_homogeneous_cube(n_paths=n_paths, film=8)
    sc["medium"] = sg.homogeneous_medium(1, conc=0.0, sigma_s=3.0, wall_mask=63, wall_albedo=1.0)
    sc["params"]["max_events"] = max_events
    S = Scene(sc)
    S.render(form="plain", hero=1)
    ref = S.read()["counters"]
    assert ref["events"] == n_paths * max_events
    for form in FORMS:
        S.render(form=form)
        assert S.read()["counters"] == ref, form
    S.close()


@pytest.mark.parametrize("dims", [(1, 1, 2), (5, 3, 7), (33, 17, 9)])
def test_negative_zeros_do_not_hide_a_maximum(dims):
    """-0.0 is accepted as 0; its bits are above those of every positive number."""
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    nx, ny, nz = dims
    results = []
    for zero in (0.0, -0.0):
        conc = np.full((1, nz, ny, nx), zero, np.float32)
        conc.reshape(-1)[-1] = 7.0
        sc = sg.cfg1_homogeneous_cube(n_paths=20_000, film=8)
        sc["medium"] = sg.grid_medium(conc, sigma_s=0.5)
        S = Scene(sc)
        film = S.render(form="wavefront_warp", skip_cell=1).clone()
        results.append((film, S.read()))
        S.close()
    (f, r), (f0, r0) = results
    assert r["counters"] == r0["counters"] and r["counters"]["majorant_violations"] == 0
    assert torch.equal(f, f0)
