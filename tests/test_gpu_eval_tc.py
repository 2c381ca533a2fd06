"""The evaluation's forward pass on the tensor cores (csrc/agn_api.cu,
eval_chunk_tc, and csrc/mlp_eval.cu, eval_head): one row and a few, row counts
around the column tiles, rows past one chunk, narrow output layers of every
kernel size and a wide one, both precisions of the handle (theta~ is fp32 in
either).  Against float64 numpy on the rows of the seeded generator: every
operand is the exact sum of three bf16 pieces and products below 2^-25 are
dropped, so a logit is within K 2^-24 of its largest partial sum and the mean
loss within 2e-6; predictions equal where the top two logits differ by more
than 1e-4."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def agn():
    import __graft_entry__ as g
    g.build()
    import paper_1710_02368_gb300 as agn
    return agn


CASES = [((8, 8, 2), 1), ((64, 48, 10), 63), ((64, 136, 4), 129), ((72, 264, 40, 16), 257),
         ((200, 1000, 1000, 10), 3001), ((64, 128, 128, 33), 700),
         ((16, 4096, 10), 12288 + 37),   # 48 Mi / 4096 rows a chunk, then 37
         ((8, 16, 3), 65536 + 5),        # 64 Ki rows uploaded at a time, then 5
         # (few rows of up to 320 inputs a layer: the CUDA cores, in any case above)
         ((328, 24, 2), 1), ((320, 136, 4), 129), ((328, 136, 4), 129), ((8, 16, 3), 8192), ((8, 16, 3), 8193),
         ((256, 256, 2), 1024), ((256, 256, 2), 1025)]


@pytest.mark.parametrize("dims,rows", CASES)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_against_float64(agn, dims, rows, prec):
    rng = np.random.default_rng(rows)
    th = np.concatenate([np.concatenate([rng.standard_normal(a * b) / np.sqrt(a),
                                         0.1 * rng.standard_normal(b)])
                         for a, b in zip(dims, dims[1:])]).astype(np.float32)
    with agn.AGN(dims, 1, 1, 0.1, 4, batch=2, n_samples=8, n_eval=rows, theta0=th,
                 precision=agn.AGN_PREC_BF16 if prec == "bf16" else agn.AGN_PREC_FP32) as h:
        loss, acc, pred = h.evaluate(with_pred=True)
        assert h.evaluate() == (loss, acc)   # the same again
    X, y, _ = agn.agn_generate_inputs(dims, agn.AGN_DIST_UNIFORM, 4, 8, rows, want_theta=False)
    z, o = X.astype(np.float64), 0
    for l, (a, b) in enumerate(zip(dims, dims[1:])):
        W, c = th[o:o + a * b].reshape(b, a), th[o + a * b:o + a * b + b]
        z = z @ W.T.astype(np.float64) + c
        if l + 2 < len(dims):
            z = np.maximum(z, 0.0)
        o += a * b + b
    mx = z.max(1)
    ref = np.mean(np.log(np.exp(z - mx[:, None]).sum(1)) + mx - z[np.arange(rows), y])
    assert abs(loss - ref) <= 2e-6 * abs(ref)
    top = np.sort(z, 1)
    clear = top[:, -1] - top[:, -2] > 1e-4
    assert np.array_equal(pred[clear], z.argmax(1)[clear])
    assert acc == pytest.approx(float(np.mean(pred == y)), abs=1e-6)


def test_cuda_core_forward_evaluates_on_the_cuda_cores(agn):
    """tc_mask without bit 0 (the forward): the evaluation's forward is the
    CUDA cores' too, bit for bit."""
    dims, out = (65536, 8, 10), []   # long sums, few samples: another order shows in the loss
    for kw in (dict(gemm=agn.AGN_GEMM_SIMT), dict(tc_mask=6)):
        with agn.AGN(dims, 1, 1, 0.1, 4, batch=2, n_samples=8, n_eval=512, **kw) as h:
            out.append(h.evaluate(with_pred=True))
    assert out[0][:2] == out[1][:2] and np.array_equal(out[0][2], out[1][2])
