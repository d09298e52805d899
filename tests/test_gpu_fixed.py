"""The FP64 form's nodal problem in 64-bit fixed point, and where it leaves
that range."""
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


# z = (b + tau eps sum) / S_nn stays below 4 at lambda 1; at lambda 2000 the
# fitting term takes some of a node's phases (or all) out of that range
@pytest.mark.parametrize("lam", [1.0, 150.0, 2000.0])
@pytest.mark.parametrize("W,H,N", [(1, 1, 2), (33, 20, 3), (64, 48, 4), (37, 23, 8)])
def test_fp64_steps_in_and_out_of_range(ac, lam, W, H, N):
    """Two steps against the oracle, both solved to 1e-13 of the data's scale:
    a step's error is at most (1 + 4 tau eps) = 33 residuals and the second
    step can raise it by 1 + 2 tau/eps = 5: 33 * 6 * 1e-13 = 2e-11, times the
    scale of z (lambda / 8 where that is above 1), whose rounding both carry."""
    img = synth.shapes_image(W + N, W, H, rect_side=(1, max(1, W // 3)), disk_r=(1, max(1.5, W / 5))).astype(np.float64)
    u0 = synth.dirichlet_init(W * N, (W + 1) * (H + 1), N)
    seg = ac.Segmenter(W, H, N, 2.0, lam, 4.0, tol=1e-13, max_cycles=2000)
    seg.set_image(img)
    seg.set_phase(u0)
    st = seg.step(2)
    assert st.converged
    u_ref, _, _ = oracle.run(img, u0, 2.0, lam, 4.0, 2, tol=1e-13, nu1=2, nu2=2)
    assert np.abs(seg.phase() - u_ref).max() < 2e-11 * max(1.0, lam / 8)
    seg.close()
