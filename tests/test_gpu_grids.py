"""The grid hierarchy of the GPU path: sides that are odd at some level."""
import numpy as np
import pytest

import oracle
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
    oracle.build()
    return mod


# odd and even sides in every combination, odd on the first level and on later
# ones, one cell more and less than the coarse tiles (32 x 16 nodes)
@pytest.mark.parametrize("W,H,N", [(9, 7, 2), (63, 33, 3), (65, 31, 4), (130, 67, 8), (126, 190, 5), (257, 102, 6),
                                   (191, 129, 8)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_odd_sides_coarsen(ac, W, H, N, precision):
    """Two steps on grids with odd sides against the oracle, with dense and
    with tiled coarse levels and with either coarse smoother.  Both sides
    solve to 1e-14 (the mixed form to 1e-13): a step's error is at most
    (1 + 4 tau eps) = 33 residuals, and the second step can raise it by
    1 + 2 tau/eps = 5, so 33 * 6 * 1e-13 = 2e-11 bounds the difference.  The
    grid levels keep the cycle count far below that of plain sweeps (about 90
    cycles to 1e-12)."""
    prec = ac.AC_MIXED if precision == "mixed" else ac.AC_FP64
    img = synth.shapes_image(W + 3 * H, W, H, rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, W / 5)))
    img64 = (synth.round_bf16(img) if precision == "mixed" else img).astype(np.float64)
    u0 = synth.dirichlet_init(W * H, (W + 1) * (H + 1), N)
    u_ref, _, _ = oracle.run(img64, u0, 2.0, 1.0, 4.0, 2, tol=1e-14, nu1=2, nu2=2)
    for tiling in (ac.AC_TILES_AUTO, ac.AC_TILES_ALWAYS):
        for smoother in (ac.AC_SMOOTH_GS3, ac.AC_SMOOTH_JACOBI):
            seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-13 if precision == "mixed" else 1e-14, max_cycles=400,
                               precision=prec)
            ac.ac_set_coarse_tiling(seg.ctx, tiling)
            ac.ac_set_coarse_smoother(seg.ctx, smoother)
            seg.set_image(img if precision == "mixed" else img64)
            seg.set_phase(u0)
            st = seg.step(2)
            assert st.total_cycles <= 90, (tiling, smoother, st.total_cycles)
            assert np.abs(seg.phase() - u_ref).max() < 2e-11, (tiling, smoother)
            seg.close()
