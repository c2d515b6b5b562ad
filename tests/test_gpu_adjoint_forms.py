"""The two forms of an orbit fit's forward pass without non-gravitational terms
-- one warp per body, with the batch midpoints inside its steps, and one lane
per body (force models the warp form does not serve: here seven corrector
iterations) -- and the backward pass over both, against the oracle's
variational gradient: one observation, many midpoints to a step, batches on the
initial epoch and before it; body counts that take a step grid with one lane per
body and stops inside its steps (from 18,000 here).  Tolerances as in test_gpu_adjoint (relative 1e-6 of loss and gradient)."""
import numpy as np
import pytest

import oracle as O
from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W
from test_gpu_adjoint import REL, _assert_grad_close, _dev, _obs_dev, _oracle_observations, _oracle_refs

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


@pytest.mark.parametrize("form", ["warp", "lane"])
@pytest.mark.parametrize("m,lo,hi,copies", [(1, 3.0, 60.0, 1), (31, 0.0, 90.0, 1), (32, -20.0, 30.0, 1),
                                            (7, 1.0, 80.0, 600),
                                            (7, 1.0, 80.0, 1000), (32, -20.0, 30.0, 1500)])
def test_gradient_matches_the_oracle(K, form, m, lo, hi, copies):
    from paper_2509_04666_gb300 import kete
    n = 18
    w = cached_workload("adjoint90", n_bodies=n, n_obs=32, neo_frac=0.2)
    rng = np.random.default_rng([m, copies])
    obs = w.meta["obs"][:, :m].copy()
    for i in range(n):
        obs["epoch"][i] = W.T0 + np.sort(rng.uniform(lo, hi, m))
    if lo < 0:
        obs["epoch"][0, ::2] = W.T0        # a batch of many on the initial epoch
        obs["epoch"][0].sort()
    orc = O.Oracle(w.ephem.to_bytes())
    fm = orc.force_model()
    obs = _oracle_observations(orc, fm, w, obs)
    y = w.states + w.meta["offsets"]
    rcs, loss_r, g_r, _ = _oracle_refs(orc, fm, y, obs)
    assert (rcs == 0).all()
    K.load_ephem(w.ephem.to_bytes())
    model = kete.force_model()
    if form == "lane":
        model.max_iter = 7
    loss, g, _, status = K.adjoint(_dev(np.tile(y, (1, copies))), _dev(np.full(n * copies, W.T0)),
                                   _obs_dev(np.tile(obs, (copies, 1))), fm=model)
    assert (status.cpu().numpy() == 0).all()
    loss, g = loss.cpu().numpy(), g.cpu().numpy()
    assert (np.abs(loss[:n] - loss_r) <= REL * loss_r).all()
    _assert_grad_close(g[:, :n], g_r)
    # every copy of a body is the same body
    assert np.array_equal(g, np.tile(g[:, :n], (1, copies)))


def test_lanes_on_the_grid_agree_with_warps(K):
    """18,000 bodies at different epochs (lanes: off the grid's points at first)
    against the same bodies 1,000 at a time (warps): loss, gradient, predictions
    and status, with a bad state, an empty row, an epoch and an observation off
    the table among them."""
    from paper_2509_04666_gb300 import kete
    n, m, copies = 1000, 6, 18
    w = cached_workload("adjoint90", n_bodies=n, n_obs=m, neo_frac=0.2)
    rng = np.random.default_rng(5)
    epochs = W.T0 + rng.uniform(-4.0, 6.0, n)
    epochs[::7] = W.T0
    obs = w.meta["obs"].copy()
    obs["ra"], obs["dec"] = rng.uniform(0.0, 6.28, (n, m)), rng.uniform(-1.0, 1.0, (n, m))
    y = w.states + w.meta["offsets"]
    y[4, 11] = np.nan
    obs["epoch"][12, :] = np.nan
    obs["epoch"][13, 3:] = np.nan
    obs["epoch"][14, -1] = W.T0 + 5000.0
    epochs[15] = W.T0 - 5000.0
    obs["epoch"][15, :] = np.nan
    K.load_ephem(w.ephem.to_bytes())

    def run(c):
        out = K.adjoint(_dev(np.tile(y, (1, c))), _dev(np.tile(epochs, c)),
                        _obs_dev(np.tile(obs, (c, 1))), pred=True)
        return [t.cpu().numpy() for t in out]

    loss, g, pred, status = run(copies)
    loss1, g1, pred1, status1 = run(1)
    assert np.array_equal(status, np.tile(status1, copies))
    assert status1[11] == kete.BODY_NONFINITE and status1[14] == status1[15] == kete.BODY_OUT_OF_SPAN
    assert (np.delete(status1, [11, 14, 15]) == 0).all()
    ok = status1 == 0
    assert np.array_equal(np.isnan(loss[:n]), np.isnan(loss1))
    assert (np.abs(loss[:n] - loss1)[ok] <= REL * loss1[ok]).all()
    assert np.array_equal(np.isnan(pred[:n]), np.isnan(pred1))
    _assert_grad_close(g[:, :n], g1, mask=ok & np.isfinite(obs["epoch"][:, 0]))
    assert np.array_equal(g, np.tile(g[:, :n], (1, copies)), equal_nan=True)
