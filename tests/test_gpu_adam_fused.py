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


@pytest.mark.parametrize("elide", [0, 1])
@pytest.mark.parametrize("prec,m", [("bf16", 33), ("fp32", 33), ("fp32", 100)])
def test_large_waves_take_the_same_steps(agn, prec, m, elide):
    """Eight workers in one wave (over 64 MB; without accumulators in bf16 mode and
    up to 96 samples Adam's own kernel) and the same shards as two waves of four
    (fused), both without split K and with the output layer's own kernel: the same
    products and sums, so the steps differ by the two kernels' contraction of the
    moments' products (2^-24 of theta_k a step; the bound leaves room for a ReLU
    decision or a bf16 rounding that this flips)."""
    dims, lam = (1024, 2056, 10), 3
    rng = np.random.default_rng(3)
    S = 2 * m + 1
    x = rng.random((8 * S, dims[0]), dtype=np.float32)
    y = rng.integers(0, 10, 8 * S).astype(np.int32)
    th0 = I.init_params(5, dims)

    def run(first, n):
        with agn.AGN(dims, n, lam, 1e-3, 5, batch=m, n_samples=n * S, theta0=th0, elide_accumulator=elide,
                     x=x[first * S:(first + n) * S], y=y[first * S:(first + n) * S],
                     precision=agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32,
                     local_optimizer=agn.AGN_OPT_ADAM, tc_mask=48) as h:
            w = np.arange(n, dtype=np.int32)
            h.run(n, w, w)   # commit k of worker k, all from version 0
            return [h.replica(k).astype(np.float64) - th0 for k in range(n)]
    for g, r in zip(run(0, 8), run(0, 4) + run(4, 4)):
        assert np.linalg.norm(g - r) <= 1e-3 * np.linalg.norm(r)
