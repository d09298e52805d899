"""Settled tiles: cycles and outer passes that visit the tiles that can change
give the numbers of those that visit every node."""
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


def _formed(W, H, N, seed):
    """Voronoi regions of pure phases with interfaces a few nodes wide; some
    nodes carry a phase of 1e-40 (no float head, no exact zero)."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H + 1, 0:W + 1]
    d = np.stack([np.hypot(x - rng.uniform(0, W), y - rng.uniform(0, H)) for _ in range(N)], -1)
    z = -d / 8.0
    s = np.sort(z, -1)[..., ::-1]
    k = np.arange(1, N + 1)
    t = (np.cumsum(s, -1) - 1) / k
    rho = (s > t).sum(-1)
    u = np.maximum(z - np.take_along_axis(t, rho[..., None] - 1, -1), 0).reshape(-1, N)
    u /= u.sum(1, keepdims=True)
    pick = rng.uniform(size=u.shape[0]) < 0.01
    u[pick, rng.integers(0, N, pick.sum())] += 1e-40
    return u


# sides at the edges of the 8-node tiles and of the coarse tiles; schedules
# whose cycles take 4 to 8 passes, the most that a tile's width allows, and 10
# (which visits every node)
@pytest.mark.parametrize("W,H,N,nu1,nu2", [(7, 9, 2, 2, 2), (63, 64, 3, 2, 1), (65, 40, 8, 2, 2), (191, 129, 4, 1, 1),
                                           (256, 130, 5, 3, 1), (130, 71, 6, 3, 2), (97, 160, 7, 0, 2)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_settled_tiles_change_no_number(ac, W, H, N, nu1, nu2, precision):
    """Steps from formed and random fields in one context, images and fields
    changed in between, with every tile visited and with the settled ones
    left out: fields, energies, cycle counts and residuals are the same bit
    for bit; so are the labels after a last step."""
    prec = ac.AC_MIXED if precision == "mixed" else ac.AC_FP64
    img = synth.shapes_image(W + N, W, H, rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, W / 5)))
    img2 = synth.shapes_image(W + N + 1, W, H, rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, W / 5)))
    formed, other = _formed(W, H, N, 1), _formed(W, H, N, 2)
    random = synth.dirichlet_init(3, (W + 1) * (H + 1), N)
    out = []
    for mode in (ac.AC_TILES_NEVER, ac.AC_TILES_ALWAYS):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-12, max_cycles=2000, precision=prec, nu1=nu1, nu2=nu2)
        ac.ac_set_coarse_tiling(seg.ctx, mode)
        seg.set_image(img)
        got = []
        for u0, image in ((formed, None), (random, None), (other, img2), (formed, None)):
            if image is not None:
                seg.set_image(image)
            seg.set_phase(u0)
            for _ in range(2):
                st = seg.step(2)
                got.append((seg.phase(), st.energy, st.residual, st.total_cycles, st.outer, seg.residual()))
        got.append((seg.segment(1),))
        out.append(got)
        seg.close()
    for a, b in zip(*out):
        assert np.array_equal(a[0], b[0])
        assert a[1:] == b[1:]


def test_settled_record_survives_the_device_loop(ac):
    """A context that changes between the loops (host with a record of its
    tiles, device without) gives the numbers of the host loop alone."""
    import torch
    W, H, N = 96, 64, 4
    img = synth.shapes_image(5, W, H, rect_side=(4, 30), disk_r=(3, 12))
    formed = _formed(W, H, N, 4)
    st = torch.cuda.Stream()
    out = []
    for switch in (False, True):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-12, max_cycles=2000, precision=ac.AC_MIXED,
                           stream=st.cuda_stream)
        seg.set_image(img)
        seg.set_phase(formed)
        for k in range(6):
            device = switch and k % 2 == 1
            ac.ac_set_coarse_tiling(seg.ctx, ac.AC_TILES_NEVER if device else ac.AC_TILES_ALWAYS)
            seg.set_cycle_loop(ac.AC_LOOP_AUTO if device else ac.AC_LOOP_HOST)
            assert seg.loop_on_device() == device
            seg.step(1)
        out.append(seg.phase())
        seg.close()
    assert np.array_equal(out[0], out[1])
