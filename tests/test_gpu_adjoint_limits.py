"""The limits of an orbit fit over long arcs and with few attempts: what the steps
that end at every midpoint and checkpoint (force models of seven corrector
iterations take them) allow, the forms whose steps pass them allow too.  A
main-belt body's own steps are 10 to 25 days long, so with checkpoints every 8 days
each is one step: 4 years of them are 183 of the 255, 500 days of 2.2-day ones 228,
and a step cut short by a midpoint costs a few more; no leg needs more than its
first step's few attempts."""
import numpy as np
import pytest

from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W
from test_gpu_adjoint import _assert_grad_close, _dev, _obs_dev

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


@pytest.mark.parametrize("days,m,ckpt,cap,copies", [
    (1460.0, 1, 8.0, 100_000, 1), (1460.0, 5, 8.0, 100_000, 1), (500.0, 1, 2.2, 100_000, 1),
    (500.0, 1, 2.2, 100_000, 1000),
    (90.0, 1, 8.0, 5, 1), (90.0, 1, 8.0, 5, 1000)])
def test_arcs_that_fit_the_stops_are_accepted(K, days, m, ckpt, cap, copies):
    from paper_2509_04666_gb300 import kete
    n = 18
    w = cached_workload("adjoint90", n_bodies=n, n_obs=m, days=days, neo_frac=0.0)
    obs = w.meta["obs"].copy()
    # observations spread over the whole arc, a batch each
    obs["epoch"] = W.T0 + days * (np.arange(m) + 0.97) / m
    obs["ra"], obs["dec"] = 1.0, 0.1
    K.load_ephem(w.ephem.to_bytes())
    out = []
    for form, c in (("stop by stop", 1), ("own steps", copies)):
        fm = kete.force_model(max_steps=cap)
        if form == "stop by stop":
            fm.max_iter = 7
        loss, g, _, status = K.adjoint(_dev(np.tile(w.states, (1, c))), _dev(np.full(n * c, W.T0)),
                                       _obs_dev(np.tile(obs, (c, 1))), fm=fm, ckpt_days=ckpt)
        out.append((loss.cpu().numpy()[:n], g.cpu().numpy()[:, :n], status.cpu().numpy()))
    assert (out[0][2] == 0).all()
    assert (out[1][2] == 0).all(), np.unique(out[1][2], return_counts=True)
    assert (np.abs(out[1][0] - out[0][0]) <= 1e-6 * out[0][0]).all()
    _assert_grad_close(out[1][1], out[0][1])


def test_arcs_past_the_limit_are_refused(K):
    """300 checkpoints: more steps than are kept, whichever form takes them."""
    from paper_2509_04666_gb300 import kete
    w = cached_workload("adjoint90", n_bodies=18, n_obs=2, days=90.0, neo_frac=0.0)
    obs = w.meta["obs"].copy()
    obs["epoch"] = W.T0 + np.array([80.0, 89.0])
    K.load_ephem(w.ephem.to_bytes())
    for copies in (1, 1000):
        for it in (7, 12):
            _, g, _, status = K.adjoint(_dev(np.tile(w.states, (1, copies))), _dev(np.full(18 * copies, W.T0)),
                                        _obs_dev(np.tile(obs, (copies, 1))), fm=kete.force_model(max_iter=it),
                                        ckpt_days=0.3)
            assert (status.cpu().numpy() == kete.BODY_ADJ_CAP).all() and np.isnan(g.cpu().numpy()).all()
