"""The accumulators' traffic (csrc/mlp_tc_dw.cu): a commit's first local step
stores a_k = g, its last one takes a_k only when the worker pulls anew later in
the run, and nothing zeroes a_k in between.  bf16 waves with accumulators over
64 MB keep several steps' activations: theta_k stays at the base of a block of
steps and a_k comes from one launch over up to 16 of them.  Against the one-tile-per-CTA dW
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
    C = sum(calls)
    w, tau = I.make_schedule(n, C + n, tau_lo, n - 1, 5)
    out = []
    with agn.AGN(dims, n, lam, 0.05, 5, batch=m, n_samples=3 * n * m, precision=prec,
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
         # lambda 1, several hidden layers, the output layer's own kernel
         ((136, 72, 264, 40, 10), 24, 6, 1, (13, 5, 9), True, 0),
         ((64, 4096, 5), 9, 9, 1, (20, 11), True, 8),
         ((1024, 2056, 10), 40, 8, 3, (8, 9), True, 0),
         # lambda 1, over 5 M parameters: bf16 pulls without the fp32 weights, then
         # ones with them for the next call
         ((1024, 5000, 10), 16, 4, 1, (9, 6), True, 0),
         ((784, 2400, 1400, 10), 24, 3, 1, (3, 2, 3), True, 2)]


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


# (dims, m, lambda, bound): lambda a multiple of the block, not one, past 16 kept
# steps; minibatches of one k step, of more, with a remainder
KEPT = [((1000, 2104, 10), 33, 5, 1 / (33 * 5)), ((1024, 1480, 400, 10), 72, 18, 3.5e-2),
        ((1024, 2072, 10), 64, 8, 1 / (64 * 8)), ((520, 4088, 10), 200, 4, 1e-2)]


@pytest.mark.parametrize("dims,m,lam,bound", KEPT)
@pytest.mark.parametrize("elide", [0, 1])
def test_kept_steps_match_small_waves(agn, dims, m, lam, bound, elide):
    """Eight workers in one wave (over 64 MB: steps kept) against the same
    shards as two handles of four (under it: every step updates theta_k and
    a_k).  The operands are the same bf16 values until the two sums' fp32
    rounding (2^-24 of theta_k) flips the rounding of a bf16 copy, about one in
    2^15 copies a step; each flip is 2^-9 of its weight and passes through the
    remaining steps' gradients, at worst through the ReLU decision of one sample:
    a share 1 / (m lambda) of the update.  The bounds are that, or, where it is
    more, four times what eight workers and twice four differed by when every
    step updated theta_k and a_k in both (1.8e-5, 8.7e-3, 1.4e-5, 2.6e-3)."""
    rng = np.random.default_rng(7)
    S = 2 * m + 3
    x = rng.random((8 * S, dims[0]), dtype=np.float32)
    y = rng.integers(0, 10, 8 * S).astype(np.int32)
    th0 = np.concatenate([np.concatenate([rng.uniform(-1, 1, a * b) * np.sqrt(6 / (a + b)),
                                          np.zeros(b)]) for a, b in zip(dims, dims[1:])])
    th0 = th0.astype(np.float32)

    def run(first, n):
        with agn.AGN(dims, n, lam, 0.002, 5, batch=m, n_samples=n * S, theta0=th0,
                     x=x[first * S:(first + n) * S], y=y[first * S:(first + n) * S],
                     precision=agn.AGN_PREC_BF16, elide_accumulator=elide) as h:
            w = np.arange(n, dtype=np.int32)
            h.run(n, w, w)   # commit k of worker k, all from version 0
            return ([h.replica(k).astype(np.float64) - th0 for k in range(n)],
                    h.central().astype(np.float64) - th0)
    r8, c8 = run(0, 8)
    ra, ca = run(0, 4)
    rb, cb = run(4, 4)
    assert np.linalg.norm(c8 - (ca + cb)) <= bound * np.linalg.norm(c8)
    for g, r in zip(r8, ra + rb):
        assert np.linalg.norm(g - r) <= bound * np.linalg.norm(r)
