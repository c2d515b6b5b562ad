"""The two forms of the propagation -- one lane per body on the step grid, one
warp per body -- against the oracle's chain of stops, at the places where a
step and the stops inside it can go wrong: several stops inside one step, two
equal stops, a stop on the initial epoch, a chain that first runs backward,
bodies at other epochs than the first, spans longer than one grid launch,
stops past the table's end, backward targets.  Position tolerance 1e-9 AU, the
parity tolerance of the other propagation tests (both sides integrate to
~1e-13 AU)."""
import numpy as np
import pytest

import oracle as O
from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-9


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


@pytest.fixture(scope="module")
def pop():
    w = cached_workload("ragged1y", n_bodies=2000)
    idx = np.concatenate([np.nonzero(w.labels == lab)[0][:n]
                          for lab, n in ((0, 17), (1, 17), (2, 5), (3, 6), (4, 4))])
    return w, w.states[:, idx].copy()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _form(K, form, precision=0):
    from paper_2509_04666_gb300 import kete
    # an explicit attempt budget keeps a small call on the lanes: 1e6 sets
    # nobody aside, 6 sets every body aside early
    split, defer = {"warp": (0, 0), "lane": (8, 1_000_000), "aside": (8, 2)}[form]
    K.set_propagation(precision, kete.PROP_WORK_STEALING, 128, split, defer)


@pytest.fixture(autouse=True)
def _default_form(K):
    yield
    _form(K, "warp", 0)
    _form(K, "warp", 1)


CHAINS = {
    "dense": W.T0 + np.array([0.0, 0.4, 0.41, 3.0, 3.0, 9.5, 10.0, 10.001, 27.3, 60.0]),
    "backward_first": W.T0 + np.array([-12.5, -3.0, 0.2, 1.0, 40.0]),
    "long_gap": W.T0 + np.array([5.0, 360.0, 361.0]),
}


@pytest.mark.parametrize("form", ["warp", "lane", "aside"])
@pytest.mark.parametrize("chain", sorted(CHAINS))
def test_chain_matches_the_oracle(K, pop, form, chain):
    w, states = pop
    stops = CHAINS[chain]
    n = states.shape[1]
    epochs = np.full(n, W.T0)
    epochs[3::4] += 1.37          # off the grid's points
    K.load_ephem(w.ephem.to_bytes())
    _form(K, form)
    out, status = K.propagate_stops(_dev(states), _dev(epochs), stops)
    out, status = out.cpu().numpy(), status.cpu().numpy()
    if form == "aside":
        assert K.get_stats()["deferred"] > 0
    orc = O.Oracle(w.ephem.to_bytes())
    for i in range(n):
        rc, ref, _ = orc.propagate_stops(orc.force_model(), states[:, i], epochs[i], stops)
        assert rc == status[i] == 0
        assert np.abs(out[:, :3, i] - ref[:, :3]).max() < TOL, (i, chain, form)


@pytest.mark.parametrize("form", ["warp", "lane"])
@pytest.mark.parametrize("days", [-0.3, -55.0, 0.25, 1.0, 365.0])
@pytest.mark.parametrize("precision", [0, 1])
def test_single_target_matches_the_oracle(K, pop, form, days, precision):
    from paper_2509_04666_gb300 import kete
    w, states = pop
    if precision:      # FP32 planet terms: not the forced encounters (other tolerance)
        states = states[:, :45]
    n = states.shape[1]
    epochs = np.full(n, W.T0)
    epochs[1::3] -= 0.77
    K.load_ephem(w.ephem.to_bytes())
    _form(K, form, precision)
    st, ep = _dev(states), _dev(epochs)
    status = K.propagate(st, ep, W.T0 + days, fm=kete.force_model(precision=precision))
    assert (status.cpu().numpy() == 0).all() and (ep.cpu().numpy() == W.T0 + days).all()
    got = st.cpu().numpy()
    orc = O.Oracle(w.ephem.to_bytes())
    for i in range(n):
        rc, ref, *_ = orc.propagate(orc.force_model(), states[:, i], epochs[i], W.T0 + days)
        assert rc == 0 and np.abs(got[:3, i] - ref[:3]).max() < TOL, (i, form, days)


@pytest.mark.parametrize("form", ["warp", "lane"])
def test_span_longer_than_one_grid(K, form):
    """600 days: the lanes cross a mark between two launches."""
    w = W.propagation_only("long", 40, 600.0, 0, n_neo=6)
    K.load_ephem(w.ephem.to_bytes())
    _form(K, form)
    stops = W.T0 + np.array([599.0, 600.0])
    out, status = K.propagate_stops(_dev(w.states), _dev(w.epochs), stops)
    assert (status.cpu().numpy() == 0).all()
    orc = O.Oracle(w.ephem.to_bytes())
    for i in range(w.n_bodies):
        rc, ref, _ = orc.propagate_stops(orc.force_model(), w.states[:, i], W.T0, stops)
        assert rc == 0 and np.abs(out.cpu().numpy()[:, :3, i] - ref[:, :3]).max() < TOL


@pytest.mark.parametrize("form", ["warp", "lane"])
def test_stops_before_a_failure_are_kept(K, pop, form):
    """Stops past the table's end fail the body; the ones before still hold."""
    from paper_2509_04666_gb300 import kete
    w, states = pop
    states = states[:, :20]
    end = w.ephem.t_end
    stops = np.array([end - 9.0, end - 0.4, end - 0.1, end + 5.0, end + 6.0])
    epochs = np.full(20, end - 30.0)
    states = states.copy()
    K.load_ephem(w.ephem.to_bytes())
    _form(K, form)
    out, status = K.propagate_stops(_dev(states), _dev(epochs), stops)
    out, status = out.cpu().numpy(), status.cpu().numpy()
    assert (status == kete.BODY_OUT_OF_SPAN).all()
    assert np.isnan(out[3:]).all()
    orc = O.Oracle(w.ephem.to_bytes())
    for i in range(20):
        _, ref, _ = orc.propagate_stops(orc.force_model(), states[:, i], epochs[i], stops[:3])
        assert np.abs(out[:3, :3, i] - ref[:, :3]).max() < TOL
    # one target past the end: the inputs stay
    st, ep = _dev(states), _dev(epochs)
    status = K.propagate(st, ep, end + 3.0)
    assert (status.cpu().numpy() == kete.BODY_OUT_OF_SPAN).all()
    assert np.array_equal(st.cpu().numpy(), states) and (ep.cpu().numpy() == epochs).all()


@pytest.mark.parametrize("target", [1e15, -1e15])
def test_target_far_off_the_table(K, pop, target):
    """More bodies than the warp form takes, a target no grid of steps could
    reach: every body is out of span, as with few bodies, and stops on the
    table before such a stop still hold."""
    from paper_2509_04666_gb300 import kete
    w, states = pop
    many = np.tile(states[:, :20], (1, 500))
    epochs = np.full(many.shape[1], W.T0)
    K.load_ephem(w.ephem.to_bytes())
    st, ep = _dev(many), _dev(epochs)
    status = K.propagate(st, ep, target)
    assert (status.cpu().numpy() == kete.BODY_OUT_OF_SPAN).all()
    assert np.array_equal(st.cpu().numpy(), many) and (ep.cpu().numpy() == epochs).all()
    if target > 0:
        out, status = K.propagate_stops(_dev(many), _dev(epochs), np.array([W.T0 + 1.0, target]))
        out = out.cpu().numpy()
        assert (status.cpu().numpy() == kete.BODY_OUT_OF_SPAN).all() and np.isnan(out[1]).all()
        orc = O.Oracle(w.ephem.to_bytes())
        for i in range(20):
            rc, ref, _ = orc.propagate_stops(orc.force_model(), states[:, i], W.T0, [W.T0 + 1.0])
            assert rc == 0 and np.abs(out[0, :3, i] - ref[0, :3]).max() < TOL


@pytest.mark.parametrize("form", ["warp", "lane", "aside"])
@pytest.mark.parametrize("precision", [0, 1])
def test_rejected_steps(K, pop, form, precision):
    """A first step too long and a safety factor that rejects whatever overshoots:
    the rejected polynomial, cut to the new length, starts the retry; forward
    and backward from the same start."""
    from paper_2509_04666_gb300 import kete
    w, states = pop
    states = states[:, :17]            # main belt
    epochs = np.full(17, W.T0 + 20.0)
    K.load_ephem(w.ephem.to_bytes())
    _form(K, form, precision)
    fm = kete.force_model(precision=precision, dt_init=60.0, safety=0.9)
    orc = O.Oracle(w.ephem.to_bytes())
    for target in (W.T0 + 300.0, W.T0 - 40.0):
        st, ep = _dev(states), _dev(epochs)
        status = K.propagate(st, ep, target, fm=fm)
        assert (status.cpu().numpy() == 0).all()
        assert K.get_stats()["rejected"] > 0
        got = st.cpu().numpy()
        for i in range(17):
            rc, ref, *_ = orc.propagate(orc.force_model(), states[:, i], epochs[i], target)
            assert rc == 0 and np.abs(got[:3, i] - ref[:3]).max() < TOL, (i, form, target)
