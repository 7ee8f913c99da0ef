"""The persistent forms hand path ids to lanes from per-warp stocks, start their paths in the tracking step,
begin connections 32 together and put unfinished marches aside. None of it may change a result: at path counts
around the sizes of a warp, a stock and a launch, every form gives the plain form's counters, tallies and film
bit for bit (both are exact sums). A batch of media is compared with the media one by one."""
import numpy as np
import pytest
import torch

import scenegen as sg
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _cube(n):
    return sg.cfg1_homogeneous_cube(n_paths=n, film=17)


def _clear_cube(n):   # no extinction at all: every path crosses the box, nothing connects
    sc = _cube(n)
    sc["medium"] = sg.homogeneous_medium(1, conc=0.0, sigma_s=0.0)
    return sc


def _walled_cube(n):
    sc = _cube(n)
    sc["medium"] = sg.homogeneous_medium(1, conc=0.5, sigma_s=5.0, sigma_a0=0.3, wall_mask=0b011111, wall_albedo=0.9)
    return sc


def _cornell(n):
    return sg.cfg2_cornell_box(width=19, height=23, grid=21, n_paths=n)


def _sheet(n):
    return sg.cfg5_light_sheet(grid=19, width=24, height=24, n_blobs=20, n_paths=n, albedo=0.999)


def _vial(n):
    return sg.vial_scene(width=20, height=20, n_paths=n)


SCENES = {"cube": (_cube, [{}]), "clear_cube": (_clear_cube, [{}]), "walled_cube": (_walled_cube, [{}]),
          "cornell": (_cornell, [{}, {"skip_cell": 1}, {"skip_cell": 3}, {"macro_cell": 4}]), "sheet": (_sheet, [{}]),
          "vial": (_vial, [{}])}


def _same(a, fa, b, fb, what):
    assert a["counters"] == b["counters"], what
    for k in ("face", "absorbed", "emitted"):
        assert np.array_equal(a[k], b[k]), (what, k)
    assert torch.equal(fa, fb), what


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("n", [1, 31, 33, 2_047, 70_001])
def test_forms_agree_at_every_path_count(name, n):
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    make, options = SCENES[name]
    S = Scene(make(n))
    for opt in options:
        # the reference: one lane per warp works, so nothing is regrouped or shared
        one = S.render(form="wavefront", block_size=32, regroup=1, **opt).clone()
        ref = S.read()
        for kw in ({"form": "plain"}, {"form": "plain", "block_size": 32, "blocks_per_sm": 1}, {"form": "wavefront_warp"},
                   {"form": "wavefront_warp", "regroup": 3}, {"form": "wavefront_warp", "block_size": 32, "blocks_per_sm": 1}):
            f = S.render(**kw, **opt)
            _same(S.read(), f, ref, one, (name, n, kw, opt))
    S.close()


@pytest.mark.parametrize("kw", [{"max_steps": 7}, {"max_events": 3}, {"n_rr": 0}, {"analog": 1}, {"max_inelastic": 1}])
def test_ends_of_paths_agree(kw):
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    for make in (_cube, _walled_cube, _cornell):
        S = Scene(make(5_003))
        one = S.render(form="wavefront", block_size=32, regroup=1, **kw).clone()
        ref = S.read()
        for form in ("plain", "wavefront_warp"):
            f = S.render(form=form, **kw)
            _same(S.read(), f, ref, one, (form, kw))
        S.close()


@pytest.mark.parametrize("hero", [1, 2, 3, 4])
def test_hero_forms_agree(hero):
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    for make in (_cornell, _cube):
        S = Scene(make(4_099))
        one = S.render(form="plain", hero=hero).clone()
        ref = S.read()
        f = S.render(form="wavefront_warp", hero=hero)
        _same(S.read(), f, ref, one, hero)
        S.close()


@pytest.mark.parametrize("film", [16, 17, 80, 81])   # even, odd; the largest with copies of its sums, the first without
@pytest.mark.parametrize("n", [(1 << 20) - 1, 1 << 20, (1 << 20) + 33])
def test_homogeneous_kernel(n, film):
    """From 2^20 paths on the warp form of a homogeneous medium runs a kernel of its own."""
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    for medium in (None, sg.homogeneous_medium(1, conc=0.5, sigma_s=5.0, sigma_a0=0.3, wall_mask=0b011111, wall_albedo=0.9)):
        sc = sg.cfg1_homogeneous_cube(n_paths=n, film=film)
        if medium is not None:
            sc["medium"] = medium
        S = Scene(sc)
        one = S.render(form="plain").clone()
        ref = S.read()
        for kw in ({}, {"block_size": 32, "blocks_per_sm": 2}):
            f = S.render(form="wavefront_warp", **kw)
            _same(S.read(), f, ref, one, (n, film, kw))
        f = S.render(form="wavefront_warp", accumulate=True)   # the second launch adds the same sums once more
        assert torch.equal(f, one + one)
        S.close()


@pytest.mark.parametrize("value", [0.5, 255.9999847412109, 256.0, 300.0])
def test_fixed_point_of_large_weights(value):
    """Tallies are sums of round(weight 2^24): a weight on either side of 2^8, where 32 bits end. An
    uncoloured box without matter passes a source's unit weight unchanged, so the weight is made by the sum of n
    escapes; the film value of a light seen by a sensor of tiny pixels is the large single contribution."""
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    sc = sg.cfg1_homogeneous_cube(n_paths=1, film=1)
    edge = 1.0 / (value * 4.0 * np.pi) ** 0.5   # one isotropic vertex: 1 / (4 pi A_pix) = value
    sc["medium"] = sg.homogeneous_medium(1, conc=0.0, sigma_s=1e4, lo=(0.0, 0.0, 0.0), hi=(1.0, 1.0, 1.0))
    sc["sensor"] = sg.ortho_sensor(1, 1, (0.5 - edge / 2, 0.5 - edge / 2, 1.0), (edge, 0.0, 0.0), (0.0, edge, 0.0),
                                   (0.0, 0.0, 1.0))
    sc["params"]["max_events"] = 1
    S = Scene(sc)
    films = [S.render(form=f).double().cpu().numpy() for f in ("plain", "wavefront", "wavefront_warp", "wavefront_pool")]
    for f in films:
        assert np.array_equal(f, films[0])
        # one contribution of value T, T = exp(-sigma depth) in (0, 1]: exact to fp32 rounding of a few operations
        assert 0.0 < f.sum() <= value * (1.0 + 1e-5)
    S.close()


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 5, 2), (33, 17, 65), (4, 70, 9)])
def test_upload_reads_every_voxel_and_every_distance(dims):
    """The upload's maxima bound the majorant (a voxel above it would be counted) and refuse a bad value in any
    voxel; the empty-space distances change neither the film's expectation nor, in what leaps nowhere, a bit."""
    require_gpu()
    from paper_1706_03024_gb300.scene import Scene
    nx, ny, nz = dims
    rng = np.random.default_rng(nx * 100 + ny)
    n = nx * ny * nz
    for at in (0, n - 1, n // 2):
        conc = np.zeros((1, nz, ny, nx), np.float32)
        conc.reshape(-1)[at] = 7.0   # one voxel holds all the dye: the maximum is there
        sc = sg.cfg1_homogeneous_cube(n_paths=20_000, film=8)
        sc["medium"] = sg.grid_medium(conc, sigma_s=0.0)
        S = Scene(sc)
        films = []
        for kw in ({}, {"skip_cell": 1}):
            for form in ("plain", "wavefront", "wavefront_warp"):
                f = S.render(form=form, **kw).clone()
                r = S.read()
                assert r["counters"]["majorant_violations"] == 0
                films.append((f, r))
            for f, r in films[-3:]:
                assert torch.equal(f, films[-3][0]) and r["counters"] == films[-3][1]["counters"]
        # leaps draw other random numbers: the same expected escapes
        a, b = (x[1]["face"].sum() for x in (films[0], films[3]))
        assert abs(a - b) <= 6.0 * (2 * 0.25 / 20_000) ** 0.5   # weights in [0, 1]: variance at most 1/4 each
        S.close()
        for bad in (-1.0, np.nan, np.inf):
            worse = rng.uniform(0.0, 1.0, conc.shape).astype(np.float32)
            worse.reshape(-1)[at] = bad
            sc["medium"] = sg.grid_medium(worse, sigma_s=0.0)
            with pytest.raises(Exception, match="negative or non-finite"):
                Scene(sc)
