"""Where the next step's cycle loop runs follows the phase field at hand."""
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


def test_step_without_a_cycle_says_nothing_about_the_field(ac):
    """A step that its first residual accepts runs no cycle and counts no free
    nodes: the loop of the next one stays where it was."""
    import torch
    st = torch.cuda.Stream()
    W, H, N = 1024, 768, 4
    seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e6, precision=ac.AC_MIXED, stream=st.cuda_stream)
    seg.set_image(synth.shapes_image(1, W, H))
    assert seg.loop_on_device()
    for _ in range(2):
        assert seg.step(1).total_cycles == 0
        assert seg.loop_on_device()
    seg.close()


def _formed(W, H, N, seed):
    """Phases separated by interfaces a few nodes wide."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H + 1, 0:W + 1]
    z = -np.stack([np.hypot(x - rng.uniform(0, W), y - rng.uniform(0, H)) for _ in range(N)], -1) / 8.0
    s = np.sort(z, -1)[..., ::-1]
    t = (np.cumsum(s, -1) - 1) / np.arange(1, N + 1)
    u = np.maximum(z - np.take_along_axis(t, ((s > t).sum(-1) - 1)[..., None], -1), 0).reshape(-1, N)
    return u / u.sum(1, keepdims=True)


@pytest.mark.parametrize("W,H,N,precision", [(512, 384, 4, "fp64"), (1024, 768, 4, "mixed")])
def test_loop_and_form_follow_the_field_that_is_set(ac, W, H, N, precision):
    """A formed field takes the next step to the host loop and the settled
    tiles, a random one (or a new image's start) to the device loop, whatever
    the last step's field was; the numbers are those of the plain host loop,
    bit for bit."""
    import torch
    img = [synth.shapes_image(W + k, W, H) for k in range(2)]
    formed = [_formed(W, H, N, k) for k in range(2)]
    random = synth.dirichlet_init(3, (W + 1) * (H + 1), N)
    out = []
    for plain in (True, False):
        st = torch.cuda.Stream()
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-10, stream=st.cuda_stream,
                           precision=ac.AC_MIXED if precision == "mixed" else ac.AC_FP64)
        if plain:
            ac.ac_set_coarse_tiling(seg.ctx, ac.AC_TILES_NEVER)
            seg.set_cycle_loop(ac.AC_LOOP_HOST)
        seg.set_image(img[0])
        got = []
        for u0, device in ((formed[0], False), (random, True), (formed[1], False), (None, True), (formed[0], False)):
            if u0 is None:
                seg.set_image(img[1])
            else:
                seg.set_phase(u0)
            assert plain or seg.loop_on_device() == device
            for _ in range(2):
                s = seg.step(1)
                got.append((seg.phase(), s.energy, s.residual, s.total_cycles, s.outer))
        out.append(got)
        seg.close()
    for a, b in zip(*out):
        assert np.array_equal(a[0], b[0])
        assert a[1:] == b[1:]


@pytest.mark.parametrize("W,H,N", [(511, 385, 3), (512, 384, 4), (256, 255, 8)])
def test_field_buffers_of_any_alignment_and_place(ac, W, H, N):
    """A field in host memory, in device memory and one double into a device
    buffer give the same choice and the same step."""
    import torch
    formed = _formed(W, H, N, 3)
    n = formed.size
    off = torch.empty(n + 1, dtype=torch.float64, device="cuda")[1:]
    dev = torch.from_numpy(formed.reshape(-1)).cuda()
    off.copy_(dev)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-10, stream=st.cuda_stream)
    seg.set_image(synth.shapes_image(W, W, H))
    out = []
    for u0 in (np.ascontiguousarray(formed), dev, off):
        seg.set_phase(u0)
        loop = seg.loop_on_device()
        seg.step(1)
        out.append((loop, seg.phase()))
    for loop, u in out[1:]:
        assert loop == out[0][0]
        assert np.array_equal(u, out[0][1])
    seg.close()
