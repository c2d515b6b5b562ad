"""An observation made from the body's own position has no direction to speak of
but a light time of zero: the fit's prediction and loss stay finite and its
status OK, as in the oracle."""
import numpy as np
import pytest

import oracle as O
from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W
from test_gpu_adjoint import _dev, _obs_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 400])
def test_observer_on_the_body(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_04666_gb300 import build as B, kete
    B.build()
    w = cached_workload("adjoint90", n_bodies=400, n_obs=1)
    obs = w.meta["obs"][:n].copy()
    obs["epoch"] = W.T0
    obs["obs"][:, 0, :] = w.states[:3, :n].T
    orc = O.Oracle(w.ephem.to_bytes())
    for i in range(n):
        rc, _, tau = orc.apparent(w.states[:, i], W.T0, W.T0, obs["obs"][i, 0])
        assert rc == 0 and tau < 1e-15
    K = kete.Kete(0)
    K.load_ephem(w.ephem.to_bytes())
    loss, _, pred, status = K.adjoint(_dev(w.states[:, :n]), _dev(np.full(n, W.T0)), _obs_dev(obs),
                                      pred=True)
    assert (status.cpu().numpy() == kete.BODY_OK).all()
    assert torch.isfinite(loss).all() and torch.isfinite(pred).all()
    K.close()
