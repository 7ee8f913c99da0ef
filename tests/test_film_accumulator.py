"""The buffer of the film's fixed-point sums: a context that has rendered a film allocates nothing for a smaller one
(the launch can then be captured in a graph, and no captured launch loses its buffer)."""
import os
import subprocess

import pytest

import scenegen as sg
from paper_1706_03024_gb300 import build as B
from paper_1706_03024_gb300 import native as N

PROGRAM = r"""
#include <cstdio>
#include "fluoro_internal.cuh"
int main()
{
    using namespace flr;
    size_t last = 0;
    for (size_t n = 0; n < ((size_t)1 << 23); n += n < 1000 ? 1 : 997) {
        const size_t c = film_capacity(n);
        if (c < n || c < last) { std::printf("film_capacity(%zu) = %zu after %zu\n", n, c, last); return 1; }
        if (n <= FILM_COPIES_MAX_VALUES && c < n * FILM_COPIES) { std::printf("no room for copies at %zu\n", n); return 1; }
        last = c;
    }
    return 0;
}
"""


def test_capacity_never_falls_as_the_film_grows(tmp_path):
    src, exe = tmp_path / "capacity.cu", tmp_path / "capacity"
    src.write_text(PROGRAM)
    subprocess.run([B._nvcc(), "-std=c++17", *B.ARCH, "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def _use_film(S, n):
    from paper_1706_03024_gb300.scene import make_sensor
    S.sensor = sg.ortho_sensor(n, n, (0.0, 0.0, 1.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0))
    S.film = None
    N.check(N.flr_set_sensor(S.ctx, make_sensor(S.sensor)), S.ctx, "flr_set_sensor")


@pytest.mark.gpu
@pytest.mark.parametrize("large,small", [(81, 80), (86, 78), (200, 81), (300, 80), (80, 79), (17, 3)])
def test_a_smaller_film_after_a_larger_one_allocates_nothing(large, small):
    from paper_1706_03024_gb300.scene import Scene
    from tests.gpu_common import require_gpu
    require_gpu()
    S = Scene(sg.cfg1_homogeneous_cube(n_paths=2_000, film=large))
    S.render(form="wavefront_warp")
    _use_film(S, small)
    N.flr_debug_fail_alloc(1)   # the next allocation of the library would fail
    try:
        for form in ("wavefront_warp", "plain", "wavefront", "wavefront_pool"):
            assert float(S.render(form=form).sum()) > 0.0
        S.render(form="wavefront_warp", n_paths=1 << 22)
    finally:
        N.flr_debug_fail_alloc(0)
    S.close()


@pytest.mark.gpu
@pytest.mark.parametrize("film,n_paths", [(1, 2_000), (33, 2_000), (64, 1 << 22), (81, 2_000)])
def test_a_film_whose_copies_find_no_memory_renders_with_one(film, n_paths):
    """A launch needs one accumulator value a film value; the copies only make it faster."""
    from paper_1706_03024_gb300.scene import Scene
    from tests.gpu_common import require_gpu
    require_gpu()
    films = []
    for fail in (0, 1):
        S = Scene(sg.cfg1_homogeneous_cube(n_paths=n_paths, film=film))
        S.render(form="wavefront_warp", film=False)
        N.flr_debug_fail_alloc(fail)   # the accumulator with all its copies
        try:
            films.append(S.render(form="wavefront_warp").clone())
        finally:
            N.flr_debug_fail_alloc(0)
        films.append(S.render(form="wavefront_warp").clone())
        S.close()
    assert float(films[0].sum()) > 0.0
    assert all(bool((f == films[0]).all()) for f in films)
