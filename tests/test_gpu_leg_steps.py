"""kete_propagate_legs bounds the step: none passes a leg's end, also where the
proposed step is shorter than a leg.  The steps of a body of small eccentricity
e vary as r^1.5, by (1 + e)^1.5 < 1.2 about their mean s: with legs of 1.6 s every
leg takes two steps or more, where 1.6 would do without a bound."""
import numpy as np
import pytest

from paper_2509_04666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_04666_gb300 import build as B, kete
    B.build()
    k = kete.Kete(0)
    yield k
    k.close()


def _steps(K, states, epoch, target, **kw):
    import torch
    st = torch.from_numpy(np.ascontiguousarray(states)).to("cuda")
    ep = torch.full((1,), epoch, dtype=torch.float64, device="cuda")
    status = K.propagate(st, ep, target, **kw)
    assert int(status[0]) == 0 and float(ep[0]) == target
    return st.cpu().numpy(), K.get_stats()["steps"]


@pytest.mark.parametrize("sign,span", [(1.0, 400.0), (-1.0, 400.0), (1.0, 30.0)])
def test_no_step_passes_a_leg(K, sign, span):
    w = W.propagation_only("legs", 24, 400.0, 0)
    K.load_ephem(w.ephem.to_bytes())
    start = W.T0 if sign > 0 else W.T0 + 400.0
    sun = W.make_planets(w.seed)
    rel = w.states - np.concatenate([sun.pos0[0], sun.vel0[0]])[:, None]
    e = W.state_to_elements(rel[:3], rel[3:], W.GM_SUN)[1]
    quiet = np.nonzero(e < 0.12)[0][:8]
    assert len(quiet) >= 4
    for i in quiet:
        body = w.states[:, i:i + 1]
        _, free = _steps(K, body, start, start + sign * 400.0)
        leg = 1.6 * 400.0 / free
        ref, n0 = _steps(K, body, start, start + sign * span)
        got, n = _steps(K, body, start, start + sign * span, leg_days=leg)
        assert np.abs(got - ref).max() < 1e-11
        assert n >= 2 * int(span / leg), (i, free, n)


def test_more_legs_than_one_launch(K):
    """600 legs of half a day: a step per leg and no more but the first's retries."""
    w = W.propagation_only("legs", 24, 400.0, 0)
    K.load_ephem(w.ephem.to_bytes())
    ref, _ = _steps(K, w.states[:, :1], W.T0, W.T0 + 300.0)
    got, n = _steps(K, w.states[:, :1], W.T0, W.T0 + 300.0, leg_days=0.5)
    assert np.abs(got - ref).max() < 1e-11
    assert 600 <= n <= 602
