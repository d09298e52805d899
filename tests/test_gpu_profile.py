"""The profile of cycles that visit settled tiles only."""
import numpy as np
import pytest

from paper_0710_0736_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ac():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0710_0736_gb300 import build
    build.build()
    from paper_0710_0736_gb300 import ac as mod
    return mod


W, H, N = 320, 260, 4


def _profiles(ac, precision, before=0):
    """Profiles of the same steps (after `before` others) from a formed field
    with every tile visited and with the settled ones left out."""
    rng = np.random.default_rng(2)
    y, x = np.mgrid[0:H + 1, 0:W + 1]
    z = -np.stack([np.hypot(x - rng.uniform(0, W), y - rng.uniform(0, H)) for _ in range(N)], -1) / 2.0
    s = np.sort(z, -1)[..., ::-1]
    t = (np.cumsum(s, -1) - 1) / np.arange(1, N + 1)
    u0 = np.maximum(z - np.take_along_axis(t, ((s > t).sum(-1) - 1)[..., None], -1), 0).reshape(-1, N)
    out = []
    for mode in (ac.AC_TILES_NEVER, ac.AC_TILES_ALWAYS):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-10,
                           precision=ac.AC_MIXED if precision == "mixed" else ac.AC_FP64)
        ac.ac_set_coarse_tiling(seg.ctx, mode)
        seg.set_cycle_loop(ac.AC_LOOP_HOST)
        seg.set_image(synth.shapes_image(W, W, H, rect_side=(20, 80), disk_r=(10, 40)))
        seg.set_phase(u0 / u0.sum(1, keepdims=True))
        if before:
            seg.step(before)
        ac.ac_set_profiling(seg.ctx, True)
        st = seg.step(4)
        out.append((st, ac.ac_get_profile(seg.ctx)))
        seg.close()
    assert out[0][0].total_cycles == out[1][0].total_cycles
    return out[0][1], out[1][1]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_plain_launch_bytes_do_not_depend_on_the_tiles(ac, precision):
    n = (W + 1) * (H + 1) * N
    for p in _profiles(ac, precision):
        assert p.smooth_bytes_per_launch == (8.0 * n if precision == "mixed" else 12.0 * n)
        assert p.smooth_corr_extra_bytes == (2.0 * n if precision == "mixed" else 4.0 * n)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_list_launches_are_not_smoother_launches(ac, precision):
    """The same cycles run as many smoother launches, whatever they visit."""
    k = ac.PROF_CLASSES.index("smooth")
    dense, settled = _profiles(ac, precision)
    assert settled.launches[k] == dense.launches[k]
    assert 0 < settled.bytes[k] < dense.bytes[k]


def test_outer_passes_on_tiles_book_what_they_visit(ac):
    """Of a mixed step only the first outer residual visits every node (24
    bytes an unknown) once the record stands; the update and the other
    residuals visit the listed tiles."""
    k = ac.PROF_CLASSES.index("outer")
    dense, settled = _profiles(ac, "mixed", before=1)
    first = 4 * 24.0 * (W + 1) * (H + 1) * N
    assert first < settled.bytes[k] < dense.bytes[k]
