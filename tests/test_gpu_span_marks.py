"""Spans longer than one step grid (512 days) with bodies at different epochs, in
the lane form: where one launch ends and the next begins is no stop of the
caller's.  A body whose epoch lies past such a mark is not carried back to it,
and a first body whose epoch lies off the table costs the others nothing.
Against the same call in the warp form, which has no marks: both integrate to
~1e-13 AU, comets and encounters are left out, so 1e-11 AU."""
import numpy as np
import pytest

from paper_2509_04666_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11
SPAN = 800.0   # days; the table reaches from T0 - 64 to past T0 + 880


@pytest.fixture(scope="module")
def K():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_04666_gb300 import build as B, kete
    B.build()
    k = kete.Kete(0)
    yield k
    k.set_propagation(0, kete.PROP_WORK_STEALING, 128)
    k.close()


@pytest.fixture(scope="module")
def pop():
    return W.propagation_only("marks", 40, SPAN, 0, n_neo=6)


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _form(K, form):
    from paper_2509_04666_gb300 import kete
    split, defer = {"warp": (0, 0), "lane": (8, 1_000_000), "aside": (8, 2)}[form]
    K.set_propagation(0, kete.PROP_WORK_STEALING, 128, split, defer)


def _run(K, w, epochs, form, target=None, stops=None):
    _form(K, form)
    if stops is not None:
        out, status = K.propagate_stops(_dev(w.states), _dev(epochs), stops)
        return out.cpu().numpy()[:, :3], status.cpu().numpy(), K.get_stats()
    st, ep = _dev(w.states), _dev(epochs)
    status = K.propagate(st, ep, target)
    return st.cpu().numpy()[:3], status.cpu().numpy(), K.get_stats()


# epoch of the first body, of the others, target (days from T0)
CASES = {
    "first_off_the_table": (-1000.0, 0.0, 700.0),
    "others_past_the_marks": (-60.0, 790.0, 800.0),
    "others_between": (-60.0, 300.0, 800.0),
    "backward_first_off_the_table": (1400.0, 800.0, 0.0),
    "backward_others_past_the_marks": (870.0, 10.0, 0.0),
    "others_beyond_the_target": (-60.0, 850.0, 800.0),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("form", ["lane", "aside"])
@pytest.mark.parametrize("stops", [False, True])
def test_marks_move_no_body(K, pop, case, form, stops):
    from paper_2509_04666_gb300 import kete
    w = pop
    K.load_ephem(w.ephem.to_bytes())
    e0, e, target = CASES[case]
    epochs = W.T0 + np.full(w.n_bodies, e) + 0.3 * np.arange(w.n_bodies) / w.n_bodies
    epochs[0] = W.T0 + e0
    arg = dict(stops=W.T0 + np.array([target, target + 3.0])) if stops else dict(target=W.T0 + target)
    ref, ref_status, warp = _run(K, w, epochs, "warp", **arg)
    got, status, st = _run(K, w, epochs, form, **arg)
    off = not W.T0 - 64.0 <= epochs[0] <= w.ephem.t_end
    assert ref_status[0] == (kete.BODY_OUT_OF_SPAN if off else 0) and (ref_status[1:] == 0).all()
    assert np.array_equal(status, ref_status)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.nanmax(np.abs(got - ref)) < TOL
    # rounded down to the grid's lengths the lanes take more steps, not twice the way
    assert st["steps"] < 1.5 * warp["steps"] + 4 * w.n_bodies


@pytest.mark.parametrize("form", ["warp", "lane", "aside"])
def test_attempts_are_counted_over_the_whole_leg(K, pop, form):
    """max_steps bounds the attempts of one leg, whatever launches it is cut into
    and whichever form finishes it: a main-belt body makes 50 to 60 in 800 days, 30
    or more in either half of them."""
    from paper_2509_04666_gb300 import kete
    w = pop
    mb = np.nonzero(w.labels == 0)[0]
    K.load_ephem(w.ephem.to_bytes())
    for cap, want in ((40, kete.BODY_STEP_CAP), (400, 0)):
        _form(K, form)
        if form == "aside":   # (most of the attempts in the lanes, the rest in the warps)
            K.set_propagation(0, kete.PROP_WORK_STEALING, 128, 8, 25)
        st, ep = _dev(w.states[:, mb]), _dev(np.full(len(mb), W.T0 - 60.0))
        status = K.propagate(st, ep, W.T0 + 800.0, fm=kete.force_model(max_steps=cap))
        if form == "aside":
            assert K.get_stats()["deferred"] > 0
        assert (status.cpu().numpy() == want).all(), np.unique(status.cpu().numpy())
