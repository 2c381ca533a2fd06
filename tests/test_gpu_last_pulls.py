"""A standalone call writes a replica once, at its worker's last pull
(csrc/last_pulls.h): random pull lists with repeats within a commit and
across commits, against the float32 oracle that performs every pull in order;
both entry points, with and without bf16 copies, with up to 4096 workers (the
table on the stack) and more."""

import numpy as np
import pytest

import agn_inputs as I  # noqa: F401  (path set-up)
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    import torch
    import paper_1710_02368_gb300 as agn
    return agn, torch, torch.device("cuda:0")


@pytest.mark.parametrize("P,n,C,most", [(1, 1, 1, 3), (1003, 3, 7, 4), (4099, 40, 33, 9),
                                        (260, 300, 5, 200), (9, 4096, 6, 250),
                                        (6, 5000, 20, 250), (3, 40000, 2, 20)])
@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("low", [False, True])
def test_last_pull_wins(env, P, n, C, most, noalloc, low):
    agn, torch, dev = env
    rng = np.random.default_rng(P + C)
    ld = (P + 3) // 4 * 4
    theta = torch.empty(P, device=dev)
    acc = torch.empty(n, ld, device=dev)
    reps = torch.full((n, ld), 5.0, device=dev)
    repb = torch.full((n, ld), 5.0, dtype=torch.bfloat16, device=dev) if low else None
    agn.agn_fill_commit_inputs(theta, acc, None, P, ld, n, 11)
    th_h, acc_h = theta.cpu().numpy().copy(), acc[:, :P].cpu().numpy().copy()
    order = rng.integers(0, n, C).tolist()
    pulls = [rng.integers(0, n, rng.integers(0, most + 1)).tolist() for _ in range(C)]
    offs = np.cumsum([0] + [len(p) for p in pulls])
    call = agn.agn_commit_pull_noalloc if noalloc else agn.agn_commit_pull
    call(theta, acc, reps, repb, P, ld, n, order, offs, [p for ps in pulls for p in ps], 0.01, 10)
    torch.cuda.synchronize()
    t, _, r, _ = O.commit_pull_fp32(th_h, {k: acc_h[k] for k in range(n)}, order, pulls, 0.01, 10)
    assert np.array_equal(theta.cpu().numpy(), t)
    pulled = {p for ps in pulls for p in ps}
    for k in range(n):
        got = reps[k, :P].cpu()
        want = torch.from_numpy(r[k]) if k in pulled else torch.full((P,), 5.0)
        assert torch.equal(got, want), k
        if low:
            assert torch.equal(repb[k, :P].cpu(), want.to(torch.bfloat16)), k


@pytest.mark.parametrize("P", [3, 4])   # the kernel's remainder loop, its vectors
@pytest.mark.parametrize("noalloc", [False, True])
def test_worker_past_2_30_is_its_own_row(env, P, noalloc):
    """Every index below n is a worker: row 2^30 is written, row 0 is not
    (buffers of 16 GiB; only these rows are touched)."""
    agn, torch, dev = env
    n, ld = (1 << 30) + 1, 4
    acc = torch.empty(n, ld, device=dev)
    reps = torch.empty(n, ld, device=dev)
    for t in (acc, reps):
        t[0] = 5.0
        t[n - 1] = 7.0
    theta = torch.arange(4, device=dev, dtype=torch.float32)[:P].contiguous()
    call = agn.agn_commit_pull_noalloc if noalloc else agn.agn_commit_pull
    call(theta, acc, reps, None, P, ld, n, [n - 1], [0, 1], [n - 1], 0.5, 1)
    torch.cuda.synchronize()
    want = torch.arange(4, dtype=torch.float32)[:P] - 3.5
    assert torch.equal(theta.cpu(), want)
    assert torch.equal(reps[n - 1, :P].cpu(), want)
    assert torch.all(reps[0] == 5.0) and torch.all(acc[0] == 5.0)
    assert torch.all(acc[n - 1, :P] == 0.0)
    del acc, reps
    torch.cuda.empty_cache()
