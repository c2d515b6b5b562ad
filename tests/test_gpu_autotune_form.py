"""The autotuner times what a call of the whole population launches: lanes on the
step grid, which read the planets from its rows, for a population past the calls
that take one warp per body, however small the sample; warps below."""
import numpy as np
import pytest

from paper_2509_04666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,lanes", [(20_000, True), (5_000, False)])
def test_sample_takes_the_form_of_the_whole(n, lanes, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_04666_gb300 import build as B, kete
    B.build()
    w = W.propagation_only("tune", 500, 90.0, 0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    states, epochs = dev(np.tile(w.states, (1, n // 500))), dev(np.full(n, W.T0))
    K = kete.Kete(0)
    K.load_ephem(w.ephem.to_bytes())
    fm = kete.force_model(precision=precision)
    stops = W.T0 + np.array([30.0, 90.0])

    def from_rows():
        s = K.get_stats()
        return s["node_evals"] / s["force_evals"]

    picked = K.autotune(states, epochs, stops, fm=fm, max_sample=1000)
    # six of the eight variants are the automatic budget's
    tuned = from_rows()
    K.propagate_stops(states, epochs, stops, fm=fm)
    full = from_rows()
    if lanes:
        assert full > 0.9 and tuned > 0.9, (tuned, full)
    else:
        assert tuned < 0.4, tuned
        if picked[3] == 0:
            assert full == 0.0
    K.close()
