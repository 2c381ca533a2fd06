"""What a user of the AGN library has it do, as cases that can be timed and compared.

Three kinds of call cover the library's device work:

  train     `AGN.run` for the next commits of a training run, then the central
            variable (`central`) and the losses so far (`loss`): what a
            training program does between two checkpoints.
  evaluate  `AGN.evaluate` on the held-out set, with the predictions.
  commit    the parameter server's step alone, on the caller's own device
            buffers (`agn_commit_pull` or `agn_commit_pull_noalloc`).

`exact` restates Algorithm 1, Eq. 1 and Eq. 2 in float64 with torch and none of
this library's arithmetic (the held-out rows of `evaluate` are part of the
library's seeded input generator, which is where they come from there too).
"""

import math

import numpy as np
import torch

import paper_1710_02368_gb300 as agn

DEV = "cuda"
L2_BYTES = 129e6


def listed():
    return [
        # The smallest training call: a checkpoint (theta~ and losses) after
        # every four commits of a small network; launches and latency count.
        dict(name="train small fp32", kind="train", dims="784-128-10", workers=4, lam=5, batch=32,
             rows=2048, eta=0.05, tau_lo=0, tau_hi=2, commits=4, precision="fp32"),
        # The paper's own setting (Section 4): fp32, random staleness, waves of
        # a few workers each.
        dict(name="train mnist-shaped fp32", kind="train", dims="784-1000-1000-10", workers=16,
             lam=15, batch=128, rows=60000, eta=0.01, tau_lo=0, tau_hi=15, commits=64,
             precision="fp32"),
        # Wide bf16 network, large minibatches, homogeneous round robin: every
        # wave holds all the workers.
        dict(name="train wide bf16", kind="train", dims="3072-2048-2048-2048-10", workers=32,
             lam=10, batch=256, rows=16000, normal=True, eta=0.01, tau_lo=31, tau_hi=31,
             commits=32, precision="bf16"),
        # The largest: 64 replicas of a 20.9 M-parameter network.
        dict(name="train large bf16", kind="train", dims="784-4096-4096-10", workers=64, lam=10,
             batch=64, rows=40000, eta=0.01, tau_lo=63, tau_hi=63, commits=64, precision="bf16"),
        # The same network without gradient accumulators, shorter exploration.
        dict(name="train large bf16 elided", kind="train", dims="784-4096-4096-10", workers=64,
             lam=5, batch=64, rows=40000, eta=0.01, tau_lo=63, tau_hi=63, commits=64,
             precision="bf16", elide=True),
        # DynSGD commits after every step (the comparison of Section 4): commit
        # and pull weigh as much as the local steps.
        dict(name="train dynsgd lambda 1 bf16", kind="train", dims="784-4096-4096-10", workers=32,
             lam=1, batch=64, rows=40000, eta=0.001, tau_lo=0, tau_hi=31, commits=64,
             precision="bf16", dynsgd=True),
        # Adam as the local optimizer (Algorithm 1 names it).
        dict(name="train adam fp32", kind="train", dims="784-1000-1000-10", workers=16, lam=15,
             batch=128, rows=60000, eta=0.0001, tau_lo=0, tau_hi=15, commits=32,
             precision="fp32", adam=True),
        # Odd sizes everywhere: feature counts, minibatch, classes.
        dict(name="train ragged fp32", kind="train", dims="613-301-150-26", workers=8, lam=5,
             batch=100, rows=12345, eta=0.02, tau_lo=0, tau_hi=7, commits=16, precision="fp32"),
        # Large minibatches on few workers.
        dict(name="train batch 512 fp32", kind="train", dims="784-1000-1000-10", workers=4, lam=5,
             batch=512, rows=60000, eta=0.02, tau_lo=3, tau_hi=3, commits=16, precision="fp32"),
        # A point of the accuracy-versus-time curves: a held-out set of the
        # usual size.
        dict(name="evaluate", kind="evaluate", dims="784-1000-1000-10", rows=10000),
        # The parameter server's step on a large vector, a commit of every
        # worker, four pulls after each.
        dict(name="commit 16M", kind="commit", params=1 << 24, workers=64, commits=64, pulls=4,
             lam=10, eta=0.01),
        # The same step in a latency-bound loop that may not allocate: a small
        # odd vector, bf16 copies kept.
        dict(name="commit small noalloc", kind="commit", params=101770, workers=4, commits=4,
             pulls=1, lam=5, eta=0.05, bf16=True, noalloc=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train", "evaluate", "commit"])
    if kind == "commit":
        workers = _log(rng, 2, 64)
        case = dict(kind="commit", params=_log(rng, 10000, 1 << 24), workers=workers,
                    commits=rng.randint(1, 64), pulls=rng.randint(0, min(8, workers)),
                    lam=rng.randint(1, 40), eta=0.01)
        if rng.random() < 0.4:
            case["bf16"] = True
        if rng.random() < 0.4:
            case["noalloc"] = True
        return case
    odd = rng.random() < 0.35
    depth = rng.randint(1, 3)

    def width(lo, hi):
        w = _log(rng, lo, hi)
        return w if odd else max(8, w // 8 * 8)

    if kind == "evaluate":
        dims = [width(64, 2048)] + [width(64, 2048) for _ in range(depth)] + [rng.randint(2, 32)]
        return dict(kind="evaluate", dims="-".join(map(str, dims)), rows=_log(rng, 500, 12000))
    classes = rng.randint(2, 16) if rng.random() < 0.75 else rng.randint(17, 100)
    dims = [width(32, 3072)] + [width(32, 4096) for _ in range(depth)] + [classes]
    workers, lam, batch = _log(rng, 1, 64), _log(rng, 1, 20), _log(rng, 8, 512)
    lo = rng.choice([0, workers - 1])
    case = dict(kind="train", dims="-".join(map(str, dims)), workers=workers, lam=lam, batch=batch,
                rows=rng.randint(max(64, workers), 20000), eta=0.01, tau_lo=lo,
                tau_hi=workers - 1, commits=rng.randint(workers, 2 * workers),
                precision=rng.choice(["fp32", "bf16"]))
    option = rng.choice(["", "", "", "elide", "adam", "dynsgd", "unnormalised"])
    if option:
        case[option] = True
        case["eta"] = 0.0001 if option == "adam" else 0.001
    # no more than the largest listed case: fewer steps, then fewer workers.
    # Sizes that run without the tensor cores today count as more work.
    most = 3e11 if odd or batch > 256 or classes > 16 else 3e12
    while _flops(case) > most or _state_bytes(case) * case["lam"] * case["commits"] > 3e11:
        if case["lam"] > 1:
            case["lam"] = (case["lam"] + 1) // 2
        elif case["workers"] > 1:
            case["workers"] = (case["workers"] + 1) // 2
            case["tau_hi"] = case["workers"] - 1
            case["tau_lo"] = min(case["tau_lo"], case["tau_hi"])
            case["commits"] = case["workers"]
        else:
            case["batch"] = max(8, case["batch"] // 2)
            if case["batch"] == 8:
                break
    return case


# -- sizes -------------------------------------------------------------------


def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _params(dims):
    return sum(a * b + b for a, b in zip(dims, dims[1:]))


def _weights(dims):
    return sum(a * b for a, b in zip(dims, dims[1:]))


def _flops(case):
    """Forward, dX (not of the first layer) and dW of every local step."""
    d = _dims(case)
    return 2.0 * case["batch"] * (3 * _weights(d) - d[0] * d[1]) * case["lam"] * case["commits"]


def _state_bytes(case):
    """A local step's read and write of one worker's parameters and accumulator
    (with Adam the moments, in bf16 mode the low-precision copy)."""
    per = 8.0 + (0 if case.get("elide") else 8) + (16 if case.get("adam") else 0)
    return (per + (2 if case["precision"] == "bf16" else 0)) * _params(_dims(case))


def work(case):
    if case["kind"] == "commit":
        p, c = case["params"], case["commits"]
        return {"bytes": p * (8.0 + 8.0 * c + case["pulls"] * c * (6.0 if case.get("bf16") else 4.0)),
                "flops": 2.0 * p * c}
    d = _dims(case)
    p = _params(d)
    if case["kind"] == "evaluate":
        return {"bytes": 4.0 * (case["rows"] * (d[0] + 2) + p), "flops": 2.0 * case["rows"] * _weights(d)}
    # per commit: its minibatches, theta~, the accumulator and a pull; a
    # replica too large for the L2 is read and written at every local step
    c, steps = case["commits"], case["lam"] * case["commits"]
    es = 2.0 if case["precision"] == "bf16" else 4.0
    state = _state_bytes(case)
    passes = steps if state / 2 > L2_BYTES / 2 else c
    return {"bytes": steps * case["batch"] * d[0] * es + c * 20.0 * p + passes * state,
            "flops": _flops(case)}


# -- inputs ------------------------------------------------------------------


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _theta0(dims, seed):
    """Glorot-uniform weights, zero biases, in the library's flat order."""
    g = _gen(seed, 1)
    out = []
    for a, b in zip(dims, dims[1:]):
        r = math.sqrt(6.0 / (a + b))
        out.append((torch.rand(a * b, generator=g, device=DEV) * 2 - 1) * r)
        out.append(torch.zeros(b, device=DEV))
    return torch.cat(out)


def _train_inputs(case, seed):
    dims = _dims(case)
    g = _gen(seed, 2)
    shape = (case["rows"], dims[0])
    normal = bool(case.get("normal"))
    x = (torch.randn if normal else torch.rand)(shape, generator=g, device=DEV)
    # labels of a random ReLU network
    w1 = torch.randn(dims[0], 64, generator=g, device=DEV) / math.sqrt(dims[0])
    w2 = torch.randn(64, dims[-1], generator=g, device=DEV)
    y = (torch.relu((x - (0.0 if normal else 0.5)) @ w1) @ (w2 - w2.mean(0))).argmax(1)
    return x, y.to(torch.int32), _theta0(dims, seed)


def _schedule(case, seed):
    """Round robin over the workers, seeded staleness; the run repeats it (its
    length is a whole number of rounds and of passes), so that it never ends."""
    n, k = case["workers"], case["commits"]
    period = math.lcm(n, k) * max(1, 4096 // math.lcm(n, k))
    tau = np.random.RandomState(seed % (1 << 31)).randint(case["tau_lo"], case["tau_hi"] + 1, period)
    c = np.arange(period)
    tau = np.minimum(tau, np.where(c < n, c, n - 1)).astype(np.int32)
    worker = (c % n).astype(np.int32)
    more = np.arange(period + k + n) % period
    return worker[more], tau[more], period


def _commit_plan(case, seed):
    r = np.random.RandomState((seed + 3) % (1 << 31))
    n, c, pulls = case["workers"], case["commits"], case["pulls"]
    worker = np.concatenate([r.permutation(n) for _ in range(-(-c // n))])[:c].astype(np.int32)
    offsets = (np.arange(c + 1) * pulls).astype(np.int32)
    pullers = [r.permutation(n)[:pulls] for _ in range(c)]
    return worker, offsets, np.concatenate(pullers).astype(np.int32) if pulls else np.zeros(0, np.int32)


def _commit_buffers(case, seed):
    n, p = case["workers"], case["params"]
    ld = (p + 3) // 4 * 4
    g = _gen(seed, 4)
    theta = torch.randn(p, generator=g, device=DEV)
    acc = torch.empty(n, ld, device=DEV).normal_(0.0, 0.1, generator=g)
    return theta, acc, ld


def prepare(case, seed):
    if case["kind"] == "commit":
        theta, acc, ld = _commit_buffers(case, seed)
        replicas = torch.zeros_like(acc)
        replicas[:, :case["params"]] = theta
        return dict(case=case, theta=theta, acc=acc, replicas=replicas, ld=ld,
                    low=replicas.to(torch.bfloat16) if case.get("bf16") else None,
                    norm=torch.zeros(case["commits"], device=DEV), plan=_commit_plan(case, seed))
    dims = _dims(case)
    if case["kind"] == "evaluate":
        handle = agn.AGN(dims, 1, 1, 0.01, seed, n_samples=64, n_eval=case["rows"],
                         theta0=_theta0(dims, seed).cpu().numpy())
        return dict(case=case, handle=handle)
    x, y, theta0 = _train_inputs(case, seed)
    handle = agn.AGN(
        dims, case["workers"], case["lam"], case["eta"], seed,
        precision=agn.AGN_PREC_BF16 if case["precision"] == "bf16" else agn.AGN_PREC_FP32,
        batch=case["batch"], n_samples=case["rows"], x=x.cpu().numpy(), y=y.cpu().numpy(),
        theta0=theta0.cpu().numpy(), normalize=0 if case.get("unnormalised") else 1,
        commit_rule=agn.AGN_COMMIT_DYNSGD if case.get("dynsgd") else agn.AGN_COMMIT_AGN,
        elide_accumulator=1 if case.get("elide") else 0,
        local_optimizer=agn.AGN_OPT_ADAM if case.get("adam") else agn.AGN_OPT_SGD)
    worker, tau, period = _schedule(case, seed)
    return dict(case=case, handle=handle, worker=worker, tau=tau, period=period, at=0)


def run(state):
    case = state["case"]
    if case["kind"] == "commit":
        call = agn.agn_commit_pull_noalloc if case.get("noalloc") else agn.agn_commit_pull
        worker, offsets, pullers = state["plan"]
        call(state["theta"], state["acc"], state["replicas"], state["low"], case["params"],
             state["ld"], case["workers"], worker, offsets, pullers, case["eta"], case["lam"],
             1, state["norm"], torch.cuda.current_stream().cuda_stream)
        p = case["params"]
        out = {"theta": state["theta"], "acc": state["acc"][:, :p],
               "replicas": state["replicas"][:, :p], "norm": state["norm"]}
        if state["low"] is not None:
            out["replicas_bf16"] = state["low"][:, :p]
        return out
    handle = state["handle"]
    if case["kind"] == "evaluate":
        # (the accuracy is the share of the predictions that are the labels)
        loss, _, pred = handle.evaluate(with_pred=True)
        return {"loss": loss, "pred": pred}
    k, a = case["commits"], state["at"]
    b = a + k + case["workers"]   # and the next commit of every worker, to look ahead
    handle.run(k, state["worker"][a:b], state["tau"][a:b])
    state["at"] = (a + k) % state["period"]
    return {"theta": handle.central(), "loss": handle.loss()}


# -- the same in 64 bits -----------------------------------------------------


def _layers(theta, dims):
    out, o = [], 0
    for a, b in zip(dims, dims[1:]):
        out.append((theta[o:o + a * b].view(b, a), theta[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _gradient(theta, dims, x, y):
    layers = _layers(theta, dims)
    h = [x]
    for i, (w, b) in enumerate(layers):
        z = torch.addmm(b, h[-1], w.t())
        h.append(z if i + 1 == len(layers) else torch.relu_(z))
    m = x.shape[0]
    logp = torch.log_softmax(h[-1], 1)
    loss = -logp[torch.arange(m, device=x.device), y].mean()
    dz = logp.exp_()
    dz[torch.arange(m, device=x.device), y] -= 1.0
    dz /= m
    grad = torch.empty_like(theta)
    for i in range(len(layers) - 1, -1, -1):
        gw, gb = _layers(grad, dims)[i]
        torch.mm(dz.t(), h[i], out=gw)
        gb.copy_(dz.sum(0))
        if i:
            dz = torch.mm(dz, layers[i][0]) * (h[i] > 0)
    return grad, loss


def _exact_train(case, seed):
    if _flops(case) > 1.5e13:
        return None   # over 20 seconds at this card's 64-bit rate
    dims, n, lam, m, eta = _dims(case), case["workers"], case["lam"], case["batch"], case["eta"]
    x, y, theta0 = _train_inputs(case, seed)
    y = y.long()
    _, tau, _ = _schedule(case, seed)
    shard = case["rows"] // n
    versions = [theta0.double()]
    t = [0] * n
    moments = {}
    losses = []
    last = {}   # last commit that reads a version
    for c in range(case["commits"]):
        last[c - int(tau[c])] = c
    for c in range(case["commits"]):
        w, v = c % n, c - int(tau[c])
        theta = versions[v].clone()
        a = torch.zeros_like(theta)
        loss = 0.0
        for _ in range(lam):
            rows = w * shard + (t[w] * m + torch.arange(m, device=DEV)) % shard
            g, step_loss = _gradient(theta, dims, x[rows].double(), y[rows])
            loss = loss + step_loss
            t[w] += 1
            if case.get("adam"):
                m1, m2 = moments.setdefault(w, (torch.zeros_like(g), torch.zeros_like(g)))
                m1.mul_(0.9).add_(g, alpha=0.1)
                m2.mul_(0.999).addcmul_(g, g, value=0.001)
                g = -eta * (m1 / (1 - 0.9 ** t[w])) / ((m2 / (1 - 0.999 ** t[w])).sqrt() + 1e-8)
            else:
                g = g * -eta
            a += g
            theta += g
        scale = (1.0 / (int(tau[c]) + 1) if case.get("dynsgd")
                 else 1.0 if case.get("unnormalised") else 1.0 / lam)
        versions.append(versions[-1] + a * scale)
        losses.append(loss / lam)
        for u in range(c):   # versions that nothing reads any more
            if versions[u] is not None and last.get(u, -1) <= c:
                versions[u] = None
    # (in bf16 mode a loss is a mean whose operands' rounding errors cancel by
    # chance: how near it comes to 64 bits says nothing)
    loss = None if case["precision"] == "bf16" else torch.stack(losses)
    return {"theta": versions[-1], "loss": loss}


def _exact_evaluate(case, seed):
    dims = _dims(case)
    x, y, _ = agn.agn_generate_inputs(dims, agn.AGN_DIST_UNIFORM, seed, 64, case["rows"],
                                      want_theta=False)
    h = torch.from_numpy(x).to(DEV).double()
    y = torch.from_numpy(y).to(DEV).long()
    layers = _layers(_theta0(dims, seed).double(), dims)
    for i, (w, b) in enumerate(layers):
        h = torch.addmm(b, h, w.t())
        if i + 1 < len(layers):
            h = torch.relu_(h)
    loss = -torch.log_softmax(h, 1)[torch.arange(len(y), device=DEV), y].mean()
    return {"loss": float(loss), "pred": None}


def _exact_commit(case, seed):
    theta, acc, _ = _commit_buffers(case, seed)
    p = case["params"]
    theta, acc = theta.double(), acc[:, :p]
    worker, offsets, pullers = _commit_plan(case, seed)
    replicas = theta.repeat(case["workers"], 1)
    norm = []
    zero = torch.zeros(case["workers"], p, device=DEV)
    spent = set()
    for c in range(case["commits"]):
        k = int(worker[c])
        if k in spent:   # its accumulator was zeroed by its earlier commit
            delta = torch.zeros_like(theta)
        else:
            delta = acc[k].double() * -(case["eta"] / case["lam"])
        spent.add(k)
        theta = theta + delta
        norm.append(delta.norm())
        for w in pullers[offsets[c]:offsets[c + 1]]:
            replicas[int(w)] = theta
    for k in range(case["workers"]):
        if k not in spent:
            zero[k] = acc[k]
    out = {"theta": theta, "acc": zero.double(), "replicas": replicas, "norm": torch.stack(norm)}
    if case.get("bf16"):
        out["replicas_bf16"] = replicas
    return out


def exact(case, seed):
    if case["kind"] == "commit":
        return _exact_commit(case, seed)
    if case["kind"] == "evaluate":
        return _exact_evaluate(case, seed)
    return _exact_train(case, seed)


def tolerance(case):
    if case["kind"] == "commit":
        # theta~, accumulators and replicas are sums of a few rounded products
        # in a fixed order; the norms may be added in another
        return {"rel": 1e-6, "max": 4e-6}
    if case["kind"] == "evaluate":
        return {"rel": 2e-6, "differ": 2e-3}
    # Four times (theta~ and losses alike) what the tensor-core and the
    # CUDA-core kernels, which add in other orders, differ by on the listed and
    # fourteen drawn cases.  A ReLU decision at a pre-activation within rounding
    # of zero moves one sample's gradient; Adam divides by small second moments.
    if case.get("adam"):
        return {"rel": 1e-2, "max": 0.3} if case["precision"] == "bf16" else {"rel": 1.2e-3, "max": 3e-2}
    if case["precision"] == "bf16":
        return {"rel": 6e-4, "max": 4e-2}
    return {"rel": 7e-5, "max": 3e-3}
