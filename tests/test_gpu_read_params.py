"""agn_central and agn_replica pack the device's padded, aligned parameters into
the flat order on the device (csrc/commit_pull.cu, pack_kernel) and copy them
into the caller's buffer: bit for bit the initial parameters that went in,
for padded and unpadded widths, one layer and several, and a buffer long
enough for its pages to be touched by several threads."""

import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def agn():
    import __graft_entry__ as g
    g.build()
    import paper_1710_02368_gb300 as agn
    return agn


@pytest.mark.parametrize("dims", [(7, 3), (5, 9, 2), (64, 48, 10), (613, 301, 150, 26),
                                  (37, 65, 33, 13, 40), (1001, 2003, 1030, 10)])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_flat_order_round_trip(agn, dims, prec):
    P = sum(a * b + b for a, b in zip(dims, dims[1:]))
    th0 = np.random.default_rng(3).standard_normal(P).astype(np.float32)
    with agn.AGN(dims, 2, 1, 0.1, 1, batch=4, n_samples=8, theta0=th0,
                 precision=agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32) as h:
        assert np.array_equal(h.central(), th0)
        assert np.array_equal(h.replica(1), th0)
        # a longer buffer: nothing past the P parameters is written
        out = np.full(P + 3, 7.0, np.float32)
        rc = agn._lib.load().agn_central(h.h, out.ctypes.data_as(agn._lib._F32P), C.c_int64(P + 3))
        assert rc == agn.AGN_OK
        assert np.array_equal(out[:P], th0) and np.all(out[P:] == 7.0)
