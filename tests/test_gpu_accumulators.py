"""The accumulators' traffic (csrc/mlp_tc_dw.cu): a commit's first local step
stores a_k = g, its last one takes a_k only when the worker pulls anew later in
the run, nothing zeroes a_k in between, and bf16 waves with accumulators over
64 MB sum up to 16 steps' gradients in one launch.  Against the one-tile-per-CTA dW
kernel (tc_mask bit 3), which reads and writes theta_k and a_k in every local
step and leaves the zeroing to the commit: theta~, losses and the replicas at
the end, for workers that pulled and for workers that did not."""

import numpy as np
import pytest

import agn_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def agn():
    import __graft_entry__ as g
    g.build()
    import paper_1710_02368_gb300 as agn
    return agn


def _run(agn, dims, m, n, prec, mask, lam, calls, look, tau_lo):
    # (many steps: a small rate, since flipped bf16 roundings of theta_k grow)
    eta = 0.05 if lam < 10 else 0.002
    C = sum(calls)
    w, tau = I.make_schedule(n, C + n, tau_lo, n - 1, 5)
    out = []
    with agn.AGN(dims, n, lam, eta, 5, batch=m, n_samples=3 * n * m, precision=prec,
                 tc_mask=mask) as h:
        th0 = h.central()
        a = 0
        for c in calls:
            b = a + c + (n if look else 0)
            h.run(c, w[a:b], tau[a:b])
            a += c
            out.append([h.central(), *(h.replica(k) for k in range(n))])
        return th0, out, h.loss()


# (dims, m, n, lambda, commits per call, look-ahead, lowest staleness)
CASES = [((64, 48, 10), 33, 3, 1, (5, 3), True, 0),          # lambda 1: a_k only, or both
         ((784, 200, 136, 10), 100, 5, 3, (7, 4), True, 0),  # some pull within the run, some later
         ((256, 130, 26), 17, 4, 2, (8,), False, 3),         # no look-ahead: replicas keep theta_k
         ((1024, 2056, 10), 64, 8, 1, (8, 8), True, 7),      # accumulators over 64 MB
         ((1024, 2056, 10), 40, 8, 3, (8, 9), True, 0),
         # bf16, full waves: a_k from the kept steps, one block of them or two
         ((1001, 2100, 10), 33, 8, 5, (9, 7), True, 7),
         ((1024, 1480, 400, 10), 72, 8, 18, (8,), False, 7)]


@pytest.mark.parametrize("dims,m,n,lam,calls,look,tau_lo", CASES)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_against_every_step_updates(agn, dims, m, n, lam, calls, look, tau_lo, prec):
    p = agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32
    th0, got, lg = _run(agn, dims, m, n, p, 7, lam, calls, look, tau_lo)
    _, ref, lr = _run(agn, dims, m, n, p, 15, lam, calls, look, tau_lo)
    # sums of m products in another order (fp32: 2^-24 sqrt(m) of the sum), in
    # bf16 mode also a bf16 rounding of theta_k flipped by it (2^-9 of one weight)
    tol = 1e-2 if prec == "bf16" else 1e-4
    for g_call, r_call in zip(got, ref):
        for g, r in zip(g_call, r_call):
            d1, d2 = (g - th0).astype(np.float64), (r - th0).astype(np.float64)
            assert np.linalg.norm(d1 - d2) <= tol * np.linalg.norm(d2) + 1e-12
    assert np.max(np.abs(lg - lr)) <= tol * np.max(np.abs(lr))
