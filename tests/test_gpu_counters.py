"""The persistent forms count in 32-bit shared-memory words that are moved on every 16,384 rounds; the
one-thread-per-path form counts in 64 bits. Long paths in a closed box pass that line several times."""
import numpy as np
import pytest

import scenegen as sg
from tests.gpu_common import require_gpu


def closed_box(n_paths, max_events):
    sc = sg.cfg1_homogeneous_cube(n_paths=n_paths, film=8)
    sc["medium"] = sg.homogeneous_medium(1, conc=0.0, sigma_s=3.0, wall_mask=63, wall_albedo=1.0)
    sc["params"]["max_events"] = max_events
    return sc


@pytest.mark.gpu
@pytest.mark.parametrize("n_paths,max_events", [(1, 16_383), (33, 40_000), (700, 20_000)])
@pytest.mark.parametrize("film", [False, True])
def test_counters_over_many_rounds_equal_the_plain_form(n_paths, max_events, film):
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    S = Scene(closed_box(n_paths, max_events))
    S.render(form="plain", film=film)
    ref = S.read()
    assert ref["counters"]["events"] == n_paths * max_events == ref["counters"]["wall_bounces"] + ref["counters"]["scatters"]
    assert ref["counters"]["cap_hits"] == n_paths
    for form, regroup in (("wavefront_warp", 0), ("wavefront_warp", 1000), ("wavefront", 0), ("wavefront_pool", 0)):
        S.render(form=form, film=film, regroup=regroup)
        g = S.read()
        assert g["counters"] == ref["counters"], (form, regroup)
        assert np.array_equal(g["face"], ref["face"])
    S.render(form="wavefront_warp", film=film, hero=1)
    assert S.read()["counters"] == ref["counters"]
    S.close()
