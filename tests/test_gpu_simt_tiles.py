"""The CUDA-core GEMMs at the edges of their tiles (32, 64 and 128 square, k
slices of 64, 32 and 16, csrc/mlp_simt.cu): minibatches and widths one below, at and
one above a tile and the k up to which 32-square tiles take short slices, with
enough workers that each tile size is taken.  Against the float64 oracle at the
fp32 tolerances of the other parity tests, and, since every output is one chain
over k in order whatever the tile, the same worker's commit bit for bit whether it
trains alone or in a wave of many."""

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


@pytest.mark.parametrize("dims,m", [((31, 33, 5), 1), ((65, 63, 20), 31), ((129, 64, 17), 33),
                                    ((127, 128, 129, 40), 65), ((257, 129, 18), 129),
                                    ((48, 49, 5), 48), ((49, 48, 18), 49)])
def test_fp32_matches_oracle(agn, dims, m):
    n, lam, C, seed = 3, 2, 5, 23
    N = n * 2 * m + 1
    w, t = I.make_schedule(n, C + n, 0, 2, seed)
    with agn.AGN(dims, n, lam, 0.05, seed, batch=m, n_samples=N, gemm=agn.AGN_GEMM_SIMT) as h:
        th0 = h.central()
        h.run(C, w, t)
        th, loss = h.central(), h.loss()
    ds = I.SyntheticDataset(seed, dims[0], N, I.DIST_UNIFORM, (dims[0], 64, dims[-1]), N // n)
    ref = O.agn_run(O.MLP(dims), th0, n, lam, 0.05, w[:C], t[:C], ds, m, N // n)
    assert np.linalg.norm(th - ref.theta) <= 1e-5 * np.linalg.norm(ref.theta)
    assert np.allclose(loss, ref.loss, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("dims,m", [((133, 259, 18), 130), ((65, 127, 33, 17), 40)])
def test_tile_does_not_change_results(agn, dims, m, prec):
    p = agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32
    x = np.random.default_rng(1).random((2 * m, dims[0]), dtype=np.float32)
    y = (np.arange(2 * m) % dims[-1]).astype(np.int32)
    th = []
    for n in (1, 4, 64):   # every worker holds the same shard; the first one commits
        with agn.AGN(dims, n, 3, 0.05, 2, batch=m, n_samples=2 * m * n, x=np.tile(x, (n, 1)),
                     y=np.tile(y, n), precision=p, gemm=agn.AGN_GEMM_SIMT) as h:
            h.run(1 if n == 1 else n, np.arange(n, dtype=np.int32), np.arange(n, dtype=np.int32))
            th.append(h.replica(0))
    assert np.array_equal(th[0], th[1]) and np.array_equal(th[0], th[2])
