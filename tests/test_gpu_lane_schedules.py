"""The lanes of the propagation where a call takes them by itself, with the
automatic set-aside budget, and their mixed precision: calls of few bodies take
one warp per body, in FP64, and show neither."""
import numpy as np
import pytest

import oracle as O
from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W
from test_gpu_parity import MAS
from test_oracle_integrator import _earth_encounter_body

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


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("precision", [0, 1])
def test_schedules_agree_bit_for_bit(K, precision):
    from paper_2509_04666_gb300 import kete
    w = cached_workload("ragged1y", n_bodies=20_000)
    K.load_ephem(w.ephem.to_bytes())
    fm = kete.force_model(precision=precision)
    epochs = w.epochs + np.resize([0.0, 0.0, 0.37], w.n_bodies)
    epochs[0] = W.T0
    stops = W.T0 + np.array([40.0, 41.0, 120.0])
    res = []
    for kind, block, order in ((kete.PROP_STATIC, 128, False), (kete.PROP_WORK_STEALING, 64, False),
                               (kete.PROP_WORK_STEALING, 128, False), (kete.PROP_STATIC, 128, True),
                               (kete.PROP_WORK_STEALING, 128, True)):
        K.set_propagation(precision, kind, block, cost_order=order)
        out, status = K.propagate_stops(_dev(w.states), _dev(epochs), stops, fm=fm)
        st = K.get_stats()
        assert st["node_evals"] > 0 and st["deferred"] > 0
        res.append((out.cpu().numpy(), status.cpu().numpy(), st["deferred"], st["steps"]))
    K.set_propagation(precision, kete.PROP_WORK_STEALING, 128)
    for out, status, aside, steps in res[1:]:
        assert np.array_equal(out, res[0][0], equal_nan=True) and np.array_equal(status, res[0][1])
        assert (aside, steps) == res[0][2:]


def test_mixed_encounters_in_the_lanes(K, mb1k):
    """FP32 planets beyond 0.2 AU, FP64 within: Earth passes at 0.003 to 0.03 AU, and
    the forced encounters of a ragged population over a year, at the bounds of the
    mixed mode (1e-9 AU; 5e-9 AU and 1 mas from the Earth at the end of the year)."""
    from paper_2509_04666_gb300 import kete
    fm = kete.force_model(precision=kete.MIXED)
    K.set_propagation(kete.MIXED, kete.PROP_WORK_STEALING, 128, 8, 1_000_000)
    orc = O.Oracle(mb1k.ephem.to_bytes())
    K.load_ephem(mb1k.ephem.to_bytes())
    st0 = np.stack([_earth_encounter_body(orc, W.T0 + 12.0, miss=m) for m in (0.003, 0.01, 0.03)], 1)
    s, e = _dev(st0), _dev(np.full(3, W.T0))
    assert (K.propagate(s, e, W.T0 + 25.0, fm=fm).cpu().numpy() == 0).all()
    ref = orc.propagate_many(orc.force_model(), st0, np.full(3, W.T0), W.T0 + 25.0)[0]
    assert np.abs(s.cpu().numpy()[:3] - ref[:3]).max() < 1e-9
    w = cached_workload("ragged1y", n_bodies=2000)
    idx = np.concatenate([np.nonzero(w.labels == 4)[0], np.arange(0, w.n_bodies, 37)])
    states, enc = w.states[:, idx].copy(), w.labels[idx] == 4
    orc = O.Oracle(w.ephem.to_bytes())
    K.load_ephem(w.ephem.to_bytes())
    s, e = _dev(states), _dev(np.full(len(idx), W.T0))
    assert (K.propagate(s, e, W.T0 + 365.0, fm=fm).cpu().numpy() == 0).all()
    st = K.get_stats()
    assert st["node_evals"] > 0 and st["deferred"] == 0
    K.set_propagation(kete.MIXED, kete.PROP_WORK_STEALING, 128)
    ref = orc.propagate_many(orc.force_model(), states, np.full(len(idx), W.T0), W.T0 + 365.0)[0]
    d = np.abs(s.cpu().numpy()[:3] - ref[:3]).max(0)
    assert d[~enc].max() < 1e-9 and d[enc].max() < 5e-9, (d[~enc].max(), d[enc].max())
    _, earth, _ = orc.ephem(3, W.T0 + 365.0)
    sky = np.linalg.norm(s.cpu().numpy()[:3] - ref[:3], axis=0) / np.linalg.norm(ref[:3] - earth[:, None], axis=0)
    assert sky.max() < MAS, sky.max() / MAS
