"""The coarsest level of the GPU path's grid hierarchy."""
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


def _step(ac, W, H, N, eps, tau, precision, smoother, **kw):
    seg = ac.Segmenter(W, H, N, eps, 1.0, tau, tol=1e-10, max_cycles=500,
                       precision=ac.AC_MIXED if precision == "mixed" else ac.AC_FP64, **kw)
    ac.ac_set_coarse_smoother(seg.ctx, smoother)
    seg.set_image(synth.shapes_image(W + N, W, H, rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, H / 5))))
    seg.set_phase(synth.dirichlet_init(3, (W + 1) * (H + 1), N))
    st = seg.step(1)
    u = seg.phase()
    seg.close()
    return u, st


# one coarse level, above the size that the one-block tail takes: ended by
# coarse_min, and by the mass (8 tau eps = 4 h^2 on its cells of side 2)
@pytest.mark.parametrize("W,H,N,eps,tau,coarse_min", [(256, 256, 2, 5.0, 25.0, 100), (255, 200, 3, 5.0, 25.0, 60),
                                                      (600, 401, 4, 1.0, 2.0, 4)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_coarsest_level_takes_gauss_seidel(ac, W, H, N, eps, tau, coarse_min, precision):
    """The coarsest level is solved by Gauss-Seidel with either smoother, so
    with no other coarse level the choice changes nothing."""
    (u, st), (v, sv) = (_step(ac, W, H, N, eps, tau, precision, s, coarse_min=coarse_min)
                        for s in (ac.AC_SMOOTH_GS3, ac.AC_SMOOTH_JACOBI))
    assert st.converged and sv.converged
    assert st.total_cycles == sv.total_cycles
    assert np.array_equal(u, v)


# hierarchies that end before the mass dominates, by the picture's size or by
# coarse_min, with the coarsest level in the one-block tail
@pytest.mark.parametrize("W,H,N,eps,tau,coarse_min", [(16, 16, 2, 5.0, 25.0, 4), (24, 24, 8, 5.0, 25.0, 4),
                                                      (32, 16, 5, 5.0, 25.0, 4), (100, 16, 4, 5.0, 25.0, 4),
                                                      (48, 40, 3, 8.0, 64.0, 4), (128, 128, 4, 5.0, 25.0, 30)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_early_coarsest_level_is_solved(ac, W, H, N, eps, tau, coarse_min, precision):
    """20 forward Gauss-Seidel sweeps solve such a level well enough for 13 to
    16 cycles a step; with fewer passes the mixed form takes 28 to 48."""
    for smoother in (ac.AC_SMOOTH_GS3, ac.AC_SMOOTH_JACOBI):
        st = _step(ac, W, H, N, eps, tau, precision, smoother, coarse_min=coarse_min)[1]
        assert st.converged and st.total_cycles <= 18, (smoother, st.total_cycles)


@pytest.mark.parametrize("W,H,coarse_min,depths", [(128, 128, 4, (3,)), (128, 128, 1, (5, 8)), (200, 70, 2, (5, 7)),
                                                   (200, 70, 64, (1,))])
def test_coarse_min_below_the_default_gives_every_level(ac, W, H, coarse_min, depths):
    """coarse_min 1 to 3 alone decides the depth; at the default the hierarchy
    ends where the mass dominates (eps 2, tau 4: on cells of side 4).  The
    tuner reports the depth: all levels, or 5.  Either way the step is the
    same minimiser: two solves to 1e-13 differ by at most twice (1 + 4 tau eps)
    = 33 residuals."""
    N, img = 3, synth.shapes_image(5, W, H, rect_side=(8, 60), disk_r=(4, 30))
    b = ac.Batch([dict(W=W, H=H, N=N, eps=2.0, tau=4.0, lam=1.0, tol=1e-10, max_cycles=500, coarse_min=coarse_min)],
                 n_streams=1)
    b.set_image(0, img)
    assert b.tune()[0][2] in depths
    b.close()
    u0, out = synth.dirichlet_init(1, (W + 1) * (H + 1), N), []
    for cm in (4, coarse_min):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-13, max_cycles=500, coarse_min=cm)
        seg.set_image(img.astype(np.float64))
        seg.set_phase(u0)
        assert seg.step(1).converged
        out.append(seg.phase())
        seg.close()
    assert np.abs(out[0] - out[1]).max() <= 2 * 33 * 1e-13
