"""Which launches of a homogeneous medium run their own kernel (runs_homogeneous): those it is faster for. The table
holds launches measured with both kernels; the results are the same bit for bit whichever runs."""
import subprocess

import numpy as np
import pytest

import scenegen as sg
from paper_1706_03024_gb300 import build as B

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "fluoro_internal.cuh"
int main()
{
    unsigned long long n;
    int form, hero, paper, film, copies, iface, grids;
    float sigma_s, edge;
    while (std::scanf("%llu %f %f %d %d %d %d %d %d %d", &n, &sigma_s, &edge, &film, &copies, &form, &hero, &paper, &iface,
                      &grids) == 10) {
        static flr::SceneDev S;
        std::memset(&S, 0, sizeof(S));
        S.homogeneous = !grids;
        S.iface = iface;
        S.sigma_s = sigma_s;
        S.hi[0] = 0.5f * edge;
        S.lo[1] = -0.25f * edge;
        S.hi[1] = 0.75f * edge;
        std::printf("%d\n", flr::runs_homogeneous(S, form, n, hero, paper, film != 0, copies) ? 1 : 0);
    }
    return 0;
}
"""
WARP, PLAIN = 2, 0
# paths, sigma_s (1 / cm), longest edge (cm), film, copies of its sums; own kernel?
TABLE = [
    # measured slower there: short launches, thick media, thin media, no copies, fp32 additions
    (1 << 20, 20, 1, 1, 8, 0), (1 << 21, 50, 1, 1, 8, 0), (1 << 22, 100, 1, 1, 8, 0), (1 << 23, 200, 1, 1, 8, 0),
    (1 << 22, 5, 1, 1, 8, 0), (1 << 24, 2, 1, 1, 8, 0), (1 << 22, 12, 1, 1, 8, 0), (20_000_000, 0.5, 1, 1, 8, 0),
    (1 << 20, 20, 1, 1, 1, 0), (4_000_000, 20, 1, 1, 1, 0), (1 << 23, 20, 1, 1, 1, 0),
    (4_000_000, 20, 1, 1, 0, 0), (1 << 20, 20, 1, 1, 0, 0), (1 << 20, 200, 1, 0, 1, 0), (1 << 20, 5, 1, 0, 1, 0),
    # measured faster there
    (1 << 22, 20, 1, 1, 8, 1), (20_000_000, 20, 1, 1, 8, 1), (1 << 23, 50, 1, 1, 8, 1), (1 << 24, 100, 1, 1, 8, 1),
    (1 << 25, 200, 1, 1, 8, 1), (1 << 24, 20, 1, 1, 1, 1), (20_000_000, 20, 1, 1, 0, 1),
    (1 << 20, 20, 1, 0, 1, 1), (1 << 22, 200, 1, 0, 1, 1),
    # the thickness counts, not the coefficient; the borders
    (1 << 22, 2, 10, 1, 8, 1), (1 << 22, 16, 1, 1, 8, 1), (1 << 22, 15.9, 1, 1, 8, 0),
    (1 << 22, 20, 0.1, 1, 8, 0), (1 << 23, 10, 10, 1, 8, 0),
    ((1 << 22) - 1, 20, 1, 1, 8, 0), ((1 << 24) - 1, 20, 1, 1, 1, 0), ((1 << 20) - 1, 20, 1, 0, 1, 0),
]


def test_the_rule_takes_the_faster_kernel(tmp_path):
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run([B._nvcc(), "-std=c++17", *B.ARCH, "-I", B.INCLUDE, "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    rows = [(*t[:5], WARP, 0, 0, 0, 0) for t in TABLE]
    big = (20_000_000, 20, 1, 1, 8)
    others = [(*big, PLAIN, 0, 0, 0, 0), (*big, WARP, 1, 0, 0, 0), (*big, WARP, 0, 1, 0, 0), (*big, WARP, 0, 0, 1, 0),
              (*big, WARP, 0, 0, 0, 1)]
    text = "\n".join(" ".join(str(v) for v in r) for r in rows + others)
    got = [int(v) for v in subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()]
    assert got == [t[5] for t in TABLE] + [0] * len(others), [t for t, g in zip(TABLE, got) if g != t[5]]


def _walled():
    return sg.homogeneous_medium(1, conc=0.5, sigma_s=20.0, sigma_a0=0.3, wall_mask=0b011111, wall_albedo=0.9)


# either side of the rule's borders: with copies (16, 17, 80), without (81), without a film
@pytest.mark.gpu
@pytest.mark.parametrize("film,n", [(16, (1 << 22) - 1), (16, 1 << 22), (17, (1 << 22) + 33), (80, (1 << 22) + 1), (81, (1 << 24) - 1),
                                    (81, (1 << 24) + 1), (0, (1 << 20) - 1), (0, (1 << 20) + 33)])
@pytest.mark.parametrize("walls", [False, True])
def test_both_kernels_give_the_plain_forms_results(film, n, walls):
    import torch

    from paper_1706_03024_gb300.scene import Scene
    from tests.gpu_common import require_gpu
    require_gpu()
    sc = sg.cfg1_homogeneous_cube(n_paths=n, film=max(film, 8))
    if walls:
        sc["medium"] = _walled()
    S = Scene(sc)
    S.render(form="plain", film=film > 0)
    one, ref = S.film_tensor().clone(), S.read()
    for kw in ({}, {"block_size": 32, "blocks_per_sm": 2}):
        S.render(form="wavefront_warp", film=film > 0, **kw)
        got = S.read()
        assert got["counters"] == ref["counters"]
        assert all(np.array_equal(got[k], ref[k]) for k in ("face", "absorbed", "emitted"))
        assert torch.equal(S.film_tensor(), one)
    S.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(1 << 24) - 1, (1 << 24) + 1])
def test_no_allocation_entry_on_both_sides_of_the_rule(n):
    """Its film has no copies: contributions are added in fp32, k of them to a value with k roundings of 2^-24; the other
    film rounds each of them to a multiple of 2^-32."""
    import torch

    from paper_1706_03024_gb300 import native as N
    from paper_1706_03024_gb300.scene import Scene
    from tests.gpu_common import require_gpu
    from tests.test_zz_no_alloc import _noalloc
    require_gpu()
    sc = sg.cfg1_homogeneous_cube(n_paths=n, film=128)
    sc["sources"][0].update(origin=(0.0, 0.0, 1.0), eu=(1.0, 0.0, 0.0), ev=(0.0, 1.0, 0.0))   # spread over the film
    S = Scene(sc)
    want_film = S.render(form="plain").clone()
    want = S.read()
    film = torch.full_like(want_film, -1.0)
    rc, got = _noalloc(sc, None, None, n, "wavefront_warp", film)
    assert rc == N.FLR_OK
    for key in ("face", "absorbed", "emitted"):
        assert np.array_equal(got[key], want[key]), key
    assert got["counters"] == want["counters"]
    k = want["counters"]["connections"] / 128 ** 2   # per pixel, over all its values
    assert torch.allclose(film, want_film, rtol=2.0 * k * 2.0 ** -24, atol=2.0 * k * 2.0 ** -33)
    S.close()
