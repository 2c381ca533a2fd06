"""Adam's step in the dW launch's epilogue (csrc/mlp_tc_dw.cu, kDwAdam), with the
bias corrections from the host's plan: several rounds of commits of workers at
different step counts, so that the moments persist and the corrections differ
between the slots of a wave.  Widths around the tiles, one and two hidden
layers, accumulators kept and elided, against the float64 oracle at the fp32
tolerances of the other parity tests (theta~ 1e-5 relative, losses 1e-5)."""

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


@pytest.mark.parametrize("dims,m,n,lam", [((8, 8, 2), 1, 2, 1), ((64, 136, 10), 33, 3, 3),
                                          ((136, 256, 120, 16), 40, 4, 2),
                                          ((128, 1000, 10), 20, 5, 4)])
@pytest.mark.parametrize("elide", [0, 1])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_matches_oracle(agn, dims, m, n, lam, elide, prec):
    C, seed, eta = 3 * n + 1, 19, 1e-3
    N = n * 2 * m + 1
    w, t = I.make_schedule(n, C + n, 0, n - 1, seed)
    with agn.AGN(dims, n, lam, eta, seed, batch=m, n_samples=N, elide_accumulator=elide,
                 precision=agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32,
                 local_optimizer=agn.AGN_OPT_ADAM) as h:
        th0 = h.central()
        h.run(n + 1, w[:2 * n + 1], t[:2 * n + 1])   # two calls: step counts continue
        h.run(C - n - 1, w[n + 1:], t[n + 1:])
        th, loss = h.central(), h.loss()
    ds = I.SyntheticDataset(seed, dims[0], N, I.DIST_UNIFORM, (dims[0], 64, dims[-1]), N // n)
    ref = O.agn_run(O.MLP(dims), th0, n, lam, eta, w[:C], t[:C], ds, m, N // n, optimizer="adam",
                    **(dict(elide_accumulator=True) if elide else {}))
    if prec == "fp32":
        assert np.linalg.norm(th - ref.theta) <= 1e-5 * np.linalg.norm(ref.theta)
        assert np.allclose(loss, ref.loss, rtol=1e-5, atol=1e-6)
    else:
        assert np.max(np.abs(loss - ref.loss)) <= 2e-2
