"""Shapes that the explicit AGN_GEMM_TCGEN05 refuses: minibatches past 256
(on the tensor cores under AGN_GEMM_AUTO: several column tiles, the fused output
layer among them), layer widths that are not multiples of 8 and output layers
of more than 16 classes (CUDA cores, softmax over any number of classes).

Every case against the float64 oracle at the fp32 tolerances of the other
parity tests (theta~ 1e-5 relative, losses 1e-5), bf16 losses within 2e-2.
"""

import numpy as np
import pytest

import agn_inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

# dims, minibatch, workers
SHAPES = [((37, 65, 13, 7), 9, 5),           # nothing a multiple of 8
          ((3, 5, 2), 1, 2),                 # the smallest
          ((61, 130, 26), 33, 3),            # odd widths, 26 classes
          ((40, 72, 33), 17, 4),             # 33 classes
          ((24, 40, 136, 130), 40, 2),       # 130 classes: the softmax in two tiles
          ((64, 136, 10), 257, 3),           # three column tiles, one sample in the last
          ((64, 136, 10), 512, 32),          # too many tiles for the fused output layer
          ((61, 48, 40, 20), 300, 3)]        # all at once


@pytest.fixture(scope="module")
def agn():
    import __graft_entry__ as g
    g.build()
    import paper_1710_02368_gb300 as agn
    return agn


def _rel(a, b):
    return float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))


def _run(agn, dims, m, n, lam=2, C=6, seed=19, oracle=True, eta=0.05, okw=None, **kw):
    N = n * 2 * m + 1
    w, t = I.make_schedule(n, C + n, 0, 2, seed)
    with agn.AGN(dims, n, lam, eta, seed, batch=m, n_samples=N, **kw) as h:
        th0 = h.central()
        h.run(C, w, t)
        out = h.central(), h.loss(), h.replica(0)
    assert np.array_equal(th0, I.init_params(seed, dims))
    if not oracle:
        return out, None
    ds = I.SyntheticDataset(seed, dims[0], N, I.DIST_UNIFORM, (dims[0], 64, dims[-1]), N // n)
    return out, O.agn_run(O.MLP(dims), th0, n, lam, eta, w[:C], t[:C], ds, m, N // n, **(okw or {}))


@pytest.mark.parametrize("dims,m,n", SHAPES)
def test_fp32_matches_oracle(agn, dims, m, n):
    (th, loss, _), ref = _run(agn, dims, m, n)
    assert _rel(th, ref.theta) <= 1e-5
    assert np.allclose(loss, ref.loss, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("dims,m,n", SHAPES)
def test_bf16_loss_matches_oracle(agn, dims, m, n):
    (_, loss, _), ref = _run(agn, dims, m, n, precision=agn.AGN_PREC_BF16)
    assert np.max(np.abs(loss - ref.loss)) <= 2e-2


@pytest.mark.parametrize("option", ["adam", "elide", "dynsgd"])
def test_options_match_oracle(agn, option):
    kw, okw, eta = {
        "adam": (dict(local_optimizer=agn.AGN_OPT_ADAM), dict(optimizer="adam"), 1e-3),
        "elide": (dict(elide_accumulator=1), dict(elide_accumulator=True), 0.05),
        "dynsgd": (dict(commit_rule=agn.AGN_COMMIT_DYNSGD), dict(staleness_scaled=True), 0.05),
    }[option]
    (th, loss, _), ref = _run(agn, (61, 48, 40, 20), 300, 3, eta=eta, okw=okw, **kw)
    assert _rel(th, ref.theta) <= 1e-5
    assert np.allclose(loss, ref.loss, rtol=1e-5, atol=1e-6)


def test_explicit_tcgen05_still_refuses(agn):
    for dims, m in (((37, 65, 10), 8), ((64, 48, 10), 257)):
        with pytest.raises(agn.AGNError) as e:
            _run(agn, dims, m, 2, oracle=False, gemm=agn.AGN_GEMM_TCGEN05)
        assert e.value.code == agn.AGN_E_UNSUPPORTED
