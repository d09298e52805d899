"""The FP64 form's two paths through a nodal problem: binary64 on every phase,
or on the phases a float pass keeps (chosen per warp by the last cycle's free
masks)."""
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


def _formed(rng, W, H, N, ties):
    """A field of pure phases with two-phase interfaces; with ties, nodes at
    which several phases are equal, or differ by a few units in the last
    place of a float or a double."""
    n = (W + 1) * (H + 1)
    first, second = rng.integers(0, N, n), rng.integers(0, N, n)
    t = np.where(rng.uniform(size=n) < 0.3, rng.uniform(size=n), 0.0)
    u = np.zeros((n, N))
    u[np.arange(n), first] += 1 - t
    u[np.arange(n), second] += t
    if ties:
        pick = rng.uniform(size=n) < 0.3
        v = np.full((n, N), 1.0 / N) + rng.choice([0.0, 1e-16, 1e-9, 1e-7, 1e-6], size=(n, N)) / N
        u[pick] = (v / v.sum(1, keepdims=True))[pick]
    return u


# N = 2 .. 8; one node, one warp's width, odd sides, and sides past a block
@pytest.mark.parametrize("W,H,N", [(1, 1, 2), (63, 40, 3), (64, 48, 4), (37, 23, 5), (130, 9, 6), (33, 65, 7),
                                   (520, 17, 8)])
@pytest.mark.parametrize("ties", [False, True])
def test_both_paths_give_the_same_bits(ac, W, H, N, ties):
    """A step from a formed field on a new context (free masks 0: the filter)
    and on one whose masks were left by a random field (most phases free: the
    plain path in the first cycle) are bit-identical, energies and cycle
    counts too; an image of few colours makes phases tie."""
    rng = np.random.default_rng(W * 31 + N)
    img = synth.shapes_image(W + N, W, H, n_colours=2 if ties else 4, sigma=0.0 if ties else 0.05,
                             rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, W / 5))).astype(np.float64)
    u0 = _formed(rng, W, H, N, ties)
    out = []
    for warm in (False, True):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-12, max_cycles=2000)
        seg.set_image(img)
        if warm:
            seg.set_phase(synth.dirichlet_init(5, (W + 1) * (H + 1), N))
            seg.step(1)
        seg.set_phase(u0)
        st = seg.step(2)
        out.append((seg.phase(), st.energy, st.total_cycles))
        seg.close()
    (ua, ea, ca), (ub, eb, cb) = out
    assert np.array_equal(ua, ub) and ea == eb and ca == cb
    assert np.abs(ua.sum(1) - 1).max() < 1e-13 and ua.min() >= 0
