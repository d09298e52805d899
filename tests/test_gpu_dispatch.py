"""Where the next step's cycle loop runs follows the phase field at hand."""
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
