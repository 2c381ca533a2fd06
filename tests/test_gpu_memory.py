"""What agn_create does when little device memory is free (csrc/agn_api.cu).

The route of a handle follows from its sizes and the device's total memory: with
most of the memory in use, but room for everything, theta~ and the evaluation
are the same bits.  Without room for the buffers that only make it faster (the
history of kept local steps, the tensor cores' evaluation, the tensor cores past
256 samples) a handle is created without them and takes the CUDA-core or
step-by-step route, bit for bit where that route has an option of its own.

Adam keeps gradients only where its step is a kernel of its own.

Each case first measures what the handle takes, then holds all of the device's
memory but that, plus or minus some."""

import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    import torch
    import paper_1710_02368_gb300 as agn
    return agn, torch


@contextlib.contextmanager
def only_free(torch, nbytes):
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    held = torch.empty(torch.cuda.mem_get_info()[0] - int(nbytes), dtype=torch.uint8, device="cuda:0")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


def _footprint(torch, make, use):
    """Device bytes of a handle in use, its kernels loaded beforehand; its results."""
    with make() as h:
        use(h)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with make() as h:
        out = use(h)
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0], out


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def _kept(agn, mask=0):
    # 135 MB of history beside about 200 MB of everything else
    n, dims = 8, (1024, 2056, 10)
    w = np.arange(n, dtype=np.int32)

    def use(h):
        h.run(n, w, w)
        return h.central(), h.loss(), h.replica(3)
    return (lambda: agn.AGN(dims, n, 16, 0.002, 5, batch=256, n_samples=8 * 300, tc_mask=mask,
                            precision=agn.AGN_PREC_BF16)), use


def test_kept_steps_do_not_depend_on_free_memory(env):
    agn, torch = env
    make, use = _kept(agn)
    need, want = _footprint(torch, make, use)
    with only_free(torch, need + 40 * MB):
        with make() as h:
            assert _same(use(h), want)


def test_no_room_for_kept_steps(env):
    agn, torch = env
    make, use = _kept(agn)
    need, want = _footprint(torch, make, use)
    # (a tc_mask that gathers every minibatch keeps no steps either)
    plain, use_plain = _kept(agn, 64)
    _, ref = _footprint(torch, plain, use_plain)
    with only_free(torch, need - 60 * MB):
        with make() as h:
            got = use(h)
    assert _same(got, ref) and not _same(got, want)


def test_evaluation_does_not_depend_on_free_memory(env):
    agn, torch = env

    def make():   # 201 MB of pieces; long sums, few samples: another route shows in the loss
        return agn.AGN((65536, 8, 10), 1, 1, 0.1, 4, batch=2, n_samples=8, n_eval=512)

    def use(h):
        return h.evaluate(with_pred=True)
    need, want = _footprint(torch, make, use)
    # (134 MB beside it while the rows are uploaded)
    with only_free(torch, need + 200 * MB):
        with make() as h:
            assert _same(use(h), want)


def test_no_room_for_the_evaluations_pieces(env):
    agn, torch = env

    def make(gemm):
        return agn.AGN((8, 4096, 3), 1, 1, 0.1, 4, batch=2, n_samples=8, n_eval=3 * 4096, gemm=gemm)

    def use(h):
        return h.evaluate(with_pred=True)
    need, _ = _footprint(torch, lambda: make(agn.AGN_GEMM_AUTO), use)
    _, ref = _footprint(torch, lambda: make(agn.AGN_GEMM_SIMT), use)
    with only_free(torch, need - 500 * MB):   # of 805 MB: the CUDA cores take 134
        with make(agn.AGN_GEMM_AUTO) as h:
            assert _same(use(h), ref)


def test_no_room_for_long_minibatches_on_the_tensor_cores(env):
    agn, torch = env
    w = np.arange(2, dtype=np.int32)

    def make(gemm):
        return agn.AGN((784, 128, 10), 2, 2, 0.05, 4, batch=512, n_samples=60000, gemm=gemm)

    def use(h):
        h.run(2, w, w)
        return h.central(), h.loss()
    need, _ = _footprint(torch, lambda: make(agn.AGN_GEMM_AUTO), use)
    _, ref = _footprint(torch, lambda: make(agn.AGN_GEMM_SIMT), use)
    with only_free(torch, need - 200 * MB):   # of 287 MB of padded shards
        with make(agn.AGN_GEMM_AUTO) as h:
            assert _same(use(h), ref)


def test_wide_hidden_layers_take_short_chunks(env):
    """Past 12288 features a chunk is under 4096 rows (48 Mi features in all)."""
    agn, torch = env

    def make(gemm, rows):
        return agn.AGN((8, 40960, 3), 1, 1, 0.1, 4, batch=2, n_samples=8, n_eval=rows, gemm=gemm)

    def use(h):
        return h.evaluate(with_pred=True)
    small, _ = _footprint(torch, lambda: make(agn.AGN_GEMM_SIMT, 1), use)
    need, got = _footprint(torch, lambda: make(agn.AGN_GEMM_AUTO, 8193), use)
    assert need - small <= 900 * MB
    _, ref = _footprint(torch, lambda: make(agn.AGN_GEMM_SIMT, 8193), use)
    # two fp32 sums of eight products and of 40960 positive ones, in other orders
    assert got[0] == pytest.approx(ref[0], rel=1e-5)
    assert np.mean(got[2] != ref[2]) <= 1e-3


@pytest.mark.parametrize("mask,arrays", [(7, 2), (3, 3)])   # fused with dW; dW on the CUDA cores
def test_adam_keeps_gradients_only_for_its_own_kernel(env, mask, arrays):
    agn, torch = env
    n, dims = 4, (1024, 2048, 10)
    P = sum(a * b + b for a, b in zip(dims, dims[1:]))
    w = np.arange(n, dtype=np.int32)

    def make(opt):
        return agn.AGN(dims, n, 1, 1e-3, 4, batch=8, n_samples=64, tc_mask=mask, local_optimizer=opt)

    def use(h):
        h.run(n, w, w)
    sgd, _ = _footprint(torch, lambda: make(agn.AGN_OPT_SGD), use)
    adam, _ = _footprint(torch, lambda: make(agn.AGN_OPT_ADAM), use)
    assert abs(adam - sgd - arrays * 4 * n * P) <= 6 * MB   # (two MB are the device's unit)
