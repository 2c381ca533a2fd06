"""The fused output layer of the last hidden layer's split-K forward
(csrc/mlp_tc.cu, launch_tc): the other ranks' partial sums and the output
layer's scratch share the stage ring, also where equal ranges of k steps leave
fewer ranks than asked for.  13 and 14 k steps of 64 (776 to 896 inputs) with
column tiles of 256 in bf16 mode are such a case (7 ranks with up to two chunks
each do not fit); fewer k steps, one row tile and several, one column tile and
several beside it.  theta~'s update and the losses against the output layer's
own kernel (tc_mask bit 5), which adds the same bf16 products in another order."""

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


@pytest.mark.parametrize("dims", [(784, 128, 10), (776, 136, 3), (832, 40, 16), (768, 128, 10),
                                  (840, 128, 10), (24, 800, 264, 10)])
@pytest.mark.parametrize("m,n", [(129, 1), (256, 1), (256, 4), (200, 8), (300, 4), (512, 2)])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_matches_the_separate_output_layer(agn, dims, m, n, prec):
    out = []
    for mask in (0, 32):
        w, tau = I.make_schedule(n, 4 * n, n - 1, n - 1, 5)
        with agn.AGN(dims, n, 2, 0.02, 5, batch=m, n_samples=2 * n * m + 1, tc_mask=mask,
                     precision=agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32) as h:
            th0 = h.central().astype(np.float64)
            h.run(3 * n, w, tau)
            out.append((h.central() - th0, h.loss()))
    # fp32 as the other comparisons of two orders of summation; bf16: a flip of one
    # bf16 rounding (2^-9) of some activations and dZ
    tol = 1e-2 if prec == "bf16" else 1e-4
    (d, l), (dr, lr) = out
    assert np.linalg.norm(d - dr) <= tol * np.linalg.norm(dr)
    assert np.max(np.abs(l - lr)) <= tol * np.max(np.abs(lr))
