"""The record of settled tiles over what can come between two steps: the
numbers are those of cycles that visit every tile."""
import numpy as np
import pytest

from paper_0710_0736_gb300 import synth

pytestmark = pytest.mark.gpu
W, H, N = 97, 130, 4


@pytest.fixture(scope="module")
def ac():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0710_0736_gb300 import build
    build.build()
    from paper_0710_0736_gb300 import ac as mod
    return mod


def _formed(w, h, seed):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:h + 1, 0:w + 1]
    z = -np.stack([np.hypot(x - rng.uniform(0, w), y - rng.uniform(0, h)) for _ in range(N)], -1) / 6.0
    s = np.sort(z, -1)[..., ::-1]
    t = (np.cumsum(s, -1) - 1) / np.arange(1, N + 1)
    u = np.maximum(z - np.take_along_axis(t, ((s > t).sum(-1) - 1)[..., None], -1), 0).reshape(-1, N)
    return np.ascontiguousarray(u / u.sum(1, keepdims=True))


def _steps(seg, got, n=2):
    for _ in range(n):
        st = seg.step(1, allow_not_converged=True)
        got.append((seg.phase(), st.energy, st.residual, st.total_cycles, st.outer, st.converged))


@pytest.mark.parametrize("between", ["unconverged", "nonfinite", "profiling", "refined", "adjoint"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_record_over_what_comes_between_steps(ac, between, precision):
    import torch
    kw = dict(refine=1, projection=ac.AC_PROJ_NODE) if between == "refined" else {}
    img = synth.shapes_image(3, W, H, rect_side=(8, 40), disk_r=(4, 15))
    out = []
    for mode in (ac.AC_TILES_NEVER, ac.AC_TILES_ALWAYS):
        seg = ac.Segmenter(W, H, N, 2.0, 1.0, 4.0, tol=1e-11, max_cycles=3 if between == "unconverged" else 500,
                           precision=ac.AC_MIXED if precision == "mixed" else ac.AC_FP64, **kw)
        ac.ac_set_coarse_tiling(seg.ctx, mode)
        seg.set_image(img)
        a, b = (_formed(seg.Wr, seg.Hr, k) for k in range(2))
        got = []
        seg.set_phase(a)
        _steps(seg, got)
        if between == "nonfinite":
            bad = a.copy()
            bad[len(bad) // 2, 1] = np.nan
            seg.set_phase(bad)
            with pytest.raises(ac.AcError):
                seg.step(1)
        elif between == "profiling":
            ac.ac_set_profiling(seg.ctx, True)
        elif between == "adjoint":
            ac.ac_adjoint_forward(seg.ctx, 3, 2)
            g = torch.from_numpy(np.random.default_rng(7).standard_normal(a.size)).cuda()
            gi, gu = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (W * H * 3, a.size))
            torch.cuda.synchronize()
            scal = ac.ac_adjoint_backward(seg.ctx, g, gi, gu)
            assert ac.ac_adjoint_recompute_diff(seg.ctx) == 0
            got.append((gi.cpu().numpy(),) + scal)
            got.append((gu.cpu().numpy(),))
            _steps(seg, got)
        seg.set_phase(b)
        _steps(seg, got)
        out.append(got)
        seg.close()
    for p, q in zip(*out):
        assert np.array_equal(p[0], q[0])
        assert p[1:] == q[1:]
