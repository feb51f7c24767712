"""fetdpic_set_external_amplitude is refused while the context stream is being captured: a graph would
set the captured amplitude again at every replay."""
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_amplitude_is_refused_under_capture():
    import torch
    from paper_1707_04333_gb300 import fetdpic
    w = inputs.pair_plasma(8, 2, kT=0.1, wc_over_wp=0.5, seed=1)
    s = fetdpic.Simulation(w, precision="fp32", sort_interval=-1, stream=torch.cuda.Stream()).load()
    s.step(1, "boris").sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s.stream, capture_error_mode="thread_local"):
        with pytest.raises(fetdpic.FetdpicError) as ei:
            s.set_external_amplitude(0.5)
        assert ei.value.code == fetdpic.ECUDA
        s.step(1, "boris")
    with torch.cuda.stream(s.stream):
        g.replay()
    s.set_external_amplitude(0.5)
    s.step(1, "boris").sync()
    del g
    s.close()
