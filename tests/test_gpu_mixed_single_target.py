"""Mixed precision to a single target in the lanes: the node velocity is predicted
in FP64, with and without non-gravitational terms.  A body whose terms are all
zero is the same body, so both kernels give the same bits."""
import numpy as np
import pytest

from conftest import cached_workload
from paper_2509_04666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("days", [40.0, 365.0, -55.0])
def test_zero_terms_change_no_bit(days):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_04666_gb300 import build as B, kete
    B.build()
    w = cached_workload("ragged1y", n_bodies=2000)
    K = kete.Kete(0)
    K.load_ephem(w.ephem.to_bytes())
    K.set_propagation(kete.MIXED, kete.PROP_WORK_STEALING, 128, 8, 1_000_000)
    got = []
    for terms in (False, True):
        fm = kete.force_model(precision=kete.MIXED)
        if terms:
            zero = kete.nongrav_to_device(np.zeros_like(W.nongrav_params(w.labels)), "cuda")
            kete.set_nongrav(fm, zero)
        st = torch.from_numpy(w.states.copy()).to("cuda")
        ep = torch.full((w.n_bodies,), W.T0, dtype=torch.float64, device="cuda")
        status = K.propagate(st, ep, W.T0 + days, fm=fm)
        assert (status.cpu().numpy() == 0).all()
        got.append(st.cpu().numpy())
    K.close()
    assert np.array_equal(*got), (np.abs(got[0] - got[1]).max(), (got[0] != got[1]).any(0).sum())
