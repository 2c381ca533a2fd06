"""fp32 dW launches whose tiles read eight operand stages or more (minibatches
from 225) run three stages beside a shorter parameter ring
(csrc/mlp_tc_dw.cu): one below, at and past that length, a remainder in the last
stage, accumulators kept and elided, against the float64 oracle at the fp32
tolerances of the other parity tests."""

import numpy as np
import pytest

import agn_inputs as I
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def agn():
    import __graft_entry__ as g
    g.build()
    import paper_1710_02368_gb300 as agn
    return agn


@pytest.mark.parametrize("m", [224, 225, 256, 301])
@pytest.mark.parametrize("elide", [0, 1])
def test_matches_oracle(agn, m, elide):
    dims, n, lam, C, seed = (136, 264, 10), 3, 2, 6, 31
    N = n * 2 * m + 1
    w, t = I.make_schedule(n, C + n, 0, 2, seed)
    with agn.AGN(dims, n, lam, 0.05, seed, batch=m, n_samples=N, elide_accumulator=elide) as h:
        th0 = h.central()
        h.run(C, w, t)
        th, loss = h.central(), h.loss()
    ds = I.SyntheticDataset(seed, dims[0], N, I.DIST_UNIFORM, (dims[0], 64, dims[-1]), N // n)
    ref = O.agn_run(O.MLP(dims), th0, n, lam, 0.05, w[:C], t[:C], ds, m, N // n,
                    **(dict(elide_accumulator=True) if elide else {}))
    assert np.linalg.norm(th - ref.theta) <= 1e-5 * np.linalg.norm(ref.theta)
    assert np.allclose(loss, ref.loss, rtol=1e-5, atol=1e-6)
