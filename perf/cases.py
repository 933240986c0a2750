"""Performance cases of the partial-jet kernels: what a user of this package has it do.

Every case is one call of the public binding (``jet.Plan``, ``jet.LossPlan``, ``jet.Batch``) on inputs of a size that
the workloads, the tests or the paper's sweeps use (Sec. 3.1.1-3.1.2: 6x64 tanh networks, 1024-16384 collocation
points, widths 16-128, and the larger benchmark networks).  ``exact`` evaluates the same quantities in float64 with
plain torch: the derivative channels by the multivariate Faa di Bruno formula, the parameter gradient by autograd.
"""

import math

import numpy as np
import torch

from paper_2606_29702_gb300 import jet, specs

LR = 1e-3
STEP0 = 100  # the Adam steps that a running training has behind it
STORE_BUDGET = 96 << 30  # the benchmark's budget of the width-256 store schedule

# family -> input domain, outputs, residual coefficients
FAMILIES = {
    "burgers": dict(domain=((-1.0, 1.0), (0.0, 1.0)), n_out=1, coefs=dict(nu=0.01 / math.pi)),
    "allen_cahn": dict(domain=((-1.0, 1.0), (0.0, 1.0)), n_out=1, coefs=dict(eps=1e-4, k=5.0)),
    "ks": dict(domain=((0.0, 2.0 * math.pi), (0.0, 1.0)), n_out=1, coefs=dict(c1=1.0, c2=1.0, c4=1.0)),
    "ns_uvp": dict(domain=((0.0, 1.0), (0.0, 1.0)), n_out=3, coefs=dict(Re=100.0)),
    "ns_psi": dict(domain=((0.0, 1.0),) * 3, n_out=2, coefs=dict(nu=0.01)),
    "helmholtz": dict(domain=((-1.0, 1.0),) * 3, n_out=1, coefs=dict(k=4.0 * math.pi)),
}


def listed():
    def one(name, family, precision, call, width, hidden, n, store=False):
        return dict(name=name, kind="plan", family=family, precision=precision, call=call, width=width, hidden=hidden,
                    n=n, store=store)

    return [
        # the small double-precision network of a verification run: gradient, loss and residual, latency counts
        one("burgers_fp64_n1000", "burgers", "fp64", "backward", 20, 4, 1000),
        # the smallest training step of the paper's sweep over N, replay-ready (device step counter), BF16
        one("burgers_bf16_n1024", "burgers", "bf16", "train_dev", 64, 6, 1024),
        # residuals at the paper's 10000 points without a gradient: evaluation, adaptive sampling
        one("ns_uvp_fp32_forward", "ns_uvp", "fp32", "forward", 64, 6, 10000),
        # full composite losses of Sec. 3.1.1 at the paper's point counts: a training step in FP32 ...
        dict(name="burgers_loss_fp32", kind="loss", family="burgers_loss", precision="fp32", call="train", width=64,
             hidden=6, scale=1.0),
        # ... and a gradient for a user's own optimiser in BF16
        dict(name="cavity_loss_bf16", kind="loss", family="cavity_loss", precision="bf16", call="backward", width=64,
             hidden=6, scale=1.0),
        # the ordinary single-precision training step: fourth-order residual, 65536 points
        one("ks_fp32", "ks", "fp32", "train", 64, 5, 65536),
        # the split-precision form, an odd number of points, gradient only
        one("ks_bf16x3_odd", "ks", "bf16x3", "backward", 64, 5, 65521),
        # mixed third-order derivatives, 13 channels: the widest channel set
        one("ns_psi_bf16", "ns_psi", "bf16", "train", 128, 6, 262144),
        # the widest network in plain FP32 (a reference gradient), ragged
        one("helmholtz_fp32_odd", "helmholtz", "fp32", "backward", 256, 8, 16385),
        # the largest: a training step of the 3->256x8->1 network on 1048576 points, store schedule
        one("helmholtz_bf16_store", "helmholtz", "bf16", "train", 256, 8, 1048576, store=True),
        # an ensemble of 64 networks trained together, BF16, one batched launch
        dict(name="ensemble_bf16", kind="batch", precision="bf16", call="train_dev", members=64, shapes=100, cap=65536),
        # a smaller ensemble in FP32: the gradients of 16 networks
        dict(name="ensemble_fp32", kind="batch", precision="fp32", call="backward", members=16, shapes=116, cap=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "small", "small", "loss", "ks", "ns_psi", "helm32", "helm16", "batch"])
    call = rng.choice(["backward", "train", "train_dev", "backward", "train", "forward"])

    def one(family, precision, width, hidden, n, store=False):
        return dict(kind="plan", family=family, precision=precision, call=call, width=width, hidden=hidden, n=n,
                    store=store)

    if kind == "fp64":
        return one(rng.choice(["burgers", "allen_cahn"]), "fp64", rng.choice([16, 20, 32]), rng.randint(3, 6),
                   _log_int(rng, 500, 4096))
    if kind == "small":
        return one(rng.choice(["burgers", "allen_cahn", "ns_uvp"]), rng.choice(["fp32", "bf16"]),
                   rng.choice([32, 64, 128]), rng.randint(3, 8), _log_int(rng, 1024, 65536))
    if kind == "loss":
        return dict(kind="loss", family=rng.choice(["burgers_loss", "cavity_loss"]),
                    precision=rng.choice(["fp32", "bf16"]), call=call, width=64, hidden=rng.randint(4, 6),
                    scale=round(rng.uniform(0.1, 1.6), 3))
    if kind == "ks":
        return one("ks", rng.choice(["fp32", "bf16", "bf16x3"]), 64, rng.randint(3, 6), _log_int(rng, 4096, 65536))
    if kind == "ns_psi":
        return one("ns_psi", rng.choice(["bf16", "bf16x3"]), 128, rng.randint(4, 6), _log_int(rng, 8192, 262144))
    if kind == "helm32":
        return one("helmholtz", "fp32", rng.choice([128, 256]), rng.randint(4, 8), _log_int(rng, 1024, 16384))
    if kind == "helm16":
        call = rng.choice(["backward", "train"])
        return one("helmholtz", "bf16", 256, rng.randint(4, 8), _log_int(rng, 16384, 1000000), store=True)
    fp32 = rng.random() < 0.4
    return dict(kind="batch", precision="fp32" if fp32 else "bf16",
                call=rng.choice(["backward", "train_dev"]) if fp32 else "train_dev",
                members=rng.randint(4, 16 if fp32 else 64), shapes=rng.randint(100, 4000),
                cap=_log_int(rng, 4096, 16384 if fp32 else 65536))


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _members(case):
    """The networks of an ensemble as single-network cases: family, width, depth and point count of member i come
    from numpy's generator shapes + i, as in the package's ensemble workload."""
    out = []
    for i in range(case["members"]):
        rng = np.random.default_rng(case["shapes"] + i)
        width, hidden = int(rng.choice([32, 64, 128])), int(rng.integers(3, 9))
        n = int(rng.integers(2048, case["cap"] + 1))
        family = "burgers" if 2 * i < case["members"] else "allen_cahn"
        coefs = dict(nu=float(10.0 ** rng.uniform(-3.0, -1.0))) if family == "burgers" else dict(eps=1e-4, k=5.0)
        out.append(dict(kind="plan", family=family, precision=case["precision"], width=width, hidden=hidden, n=n,
                        store=False, coefs=coefs))
    return out


def _network(case):
    fam = FAMILIES["burgers" if case["kind"] == "loss" else case["family"]]
    n_out = {"burgers_loss": 1, "cavity_loss": 3}.get(case["family"], fam["n_out"])
    return [len(fam["domain"])] + [case["width"]] * case["hidden"] + [n_out]


def _loss_counts(case):
    """Points of each term, in term order."""
    s = case["scale"]
    if case["family"] == "burgers_loss":  # periodic pairs (two points each), initial condition, PDE
        return [2 * max(1, round(1000 * s)), max(1, round(101 * s)), max(1, round(10000 * s))]
    return [max(1, round(10000 * s)), max(1, round(1499 * s)), max(1, round(499 * s))]  # PDE, walls, lid


def _points(case, g):
    """(X, source or None) in float64."""
    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)

    if case["kind"] == "loss":
        a, b, c = _loss_counts(case)
        X = rand(a + b + c, 2)
        if case["family"] == "burgers_loss":
            X[0:a:2, 0], X[1:a:2, 0] = 0.0, 1.0
            X[1:a:2, 1] = X[0:a:2, 1]
            X[a:a + b, 1] = 0.0
            src = torch.zeros(X.shape[0], 2, device="cuda", dtype=torch.float64)
            src[a:a + b, 0] = -torch.sin(2.0 * math.pi * X[a:a + b, 0])
            return X, src
        side = (rand(b) * 3.0).long()
        wall = X[a:a + b]
        wall[:, 0] = torch.where(side == 0, 0.0, torch.where(side == 1, 1.0, wall[:, 0]))
        wall[:, 1] = torch.where(side == 2, 0.0, wall[:, 1])
        X[a + b:, 1] = 1.0
        src = torch.zeros(X.shape[0], 3, device="cuda", dtype=torch.float64)
        src[a + b:, 0] = 1.0
        return X, src
    domain = FAMILIES[case["family"]]["domain"]
    X = rand(case["n"], len(domain))
    for i, (lo, hi) in enumerate(domain):
        X[:, i] = lo + (hi - lo) * X[:, i]
    if case["family"] != "helmholtz":
        return X, None
    k = FAMILIES["helmholtz"]["coefs"]["k"]
    return X, (k * k - 3.0 * math.pi ** 2) * torch.sin(math.pi * X).prod(1, keepdim=True)


def _inputs(case, g):
    """Points, source, packed parameters (Xavier-normal weights, small biases) and the Adam moments of a running
    training, in the form's value type."""
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    X, src = _points(case, g)
    widths, parts = _network(case), []
    for fi, fo in zip(widths[:-1], widths[1:]):
        parts.append(torch.randn(fo * fi, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(2.0 / (fi + fo)))
        parts.append(torch.randn(fo, generator=g, device="cuda", dtype=torch.float64) * 0.1)
    params = torch.cat(parts).to(dtype)
    m = (0.1 * torch.randn(params.shape[0], generator=g, device="cuda", dtype=torch.float64)).to(dtype)
    v = (0.01 + 0.01 * torch.rand(params.shape[0], generator=g, device="cuda", dtype=torch.float64)).to(dtype)
    return dict(X=X.to(dtype), source=None if src is None else src.to(dtype), params=params, m=m, v=v)


def _plan(case):
    if case["kind"] == "loss":
        terms = specs.burgers_loss_terms(0.01) if case["family"] == "burgers_loss" else specs.cavity_loss_terms(100.0)
        plan = jet.LossPlan(terms, _network(case), case["precision"])
        plan.set_term_points(_loss_counts(case))
        return plan
    spec = specs.by_name(case["family"], **case.get("coefs", FAMILIES[case["family"]]["coefs"]))
    kw = dict(store=True, mem_budget=STORE_BUDGET) if case["store"] else {}
    return jet.Plan(spec, _network(case), case["precision"], **kw)


def prepare(case, seed):
    g = _generator(seed)
    s = dict(call=case["call"], step=STEP0)
    if case["call"] == "train_dev":
        s["counter"] = torch.full((1,), STEP0, dtype=torch.int64, device="cuda")
    if case["kind"] != "batch":
        s.update(_inputs(case, g), plan=_plan(case))
        return s
    members = _members(case)
    ins = [_inputs(c, g) for c in members]
    s["X"] = [x["X"] for x in ins]
    for k in ("params", "m", "v"):  # each member's part of one buffer
        s["all_" + k] = torch.cat([x[k] for x in ins])
        s[k] = list(s["all_" + k].split([x[k].shape[0] for x in ins]))
    s["batch"] = jet.Batch([_plan(c) for c in members])
    s["batch"].backward(s["params"], s["X"])  # a program's warm-up call, as before a graph capture
    return s


def run(s):
    call = s["call"]
    if "batch" in s:
        if call == "backward":
            grads, loss = s["batch"].backward(s["params"], s["X"])
            return {"loss": loss, "grad": grads}
        loss = s["batch"].train_step_dev(s["params"], s["m"], s["v"], s["counter"], LR, s["X"])
        return {"loss": loss, "params": s["all_params"], "m": s["all_m"], "v": s["all_v"]}
    plan = s["plan"]
    if call == "forward":
        r, loss = plan.forward(s["params"], s["X"], s["source"])
        return {"r": r, "loss": loss}
    if call == "backward":
        grad, loss, r = plan.backward(s["params"], s["X"], s["source"], want_r=True)
        return {"r": r, "loss": loss, "grad": grad}
    if call == "train":
        s["step"] += 1
        loss = plan.train_step(s["params"], s["m"], s["v"], s["step"], LR, s["X"], s["source"])
    else:
        loss = plan.train_step_dev(s["params"], s["m"], s["v"], s["counter"], LR, s["X"], s["source"])
    return {"loss": loss, "params": s["params"], "m": s["m"], "v": s["v"]}


# ------------------------------------------------------------------ work
_ORDERS = {  # derivative channels of each family's closure
    "burgers": ["", "x", "t", "xx"], "allen_cahn": ["", "x", "t", "xx"],
    "ks": ["", "x", "t", "xx", "xxx", "xxxx"], "ns_uvp": ["", "x", "y", "xx", "yy"],
    "helmholtz": ["", "x", "y", "z", "xx", "yy", "zz"],
    "ns_psi": ["", "x", "y", "t", "xx", "xy", "yy", "xt", "yt", "xxx", "xxy", "xyy", "yyy"],
}
_AXES = {"burgers": "xt", "allen_cahn": "xt", "ks": "xt", "ns_uvp": "xy", "helmholtz": "xyz", "ns_psi": "xyt"}
_BASE = {"burgers_loss": "burgers", "cavity_loss": "ns_uvp"}
_N_RES = {"ns_uvp": 3, "ns_psi": 2, "burgers_loss": 2, "cavity_loss": 3}


def work(case):
    """Inputs read once, outputs written once; the jet GEMMs of the forward pass and, with a gradient, the data and
    weight gradients' (bias, activation and residual arithmetic left out)."""
    if case["kind"] == "batch":
        each = [work(dict(c, call=case["call"])) for c in _members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    elem = 8 if case["precision"] == "fp64" else 4
    widths, family = _network(case), case["family"]
    n = sum(_loss_counts(case)) if case["kind"] == "loss" else case["n"]
    n_res = _N_RES.get(family, 1)
    n_par = sum(a * b + b for a, b in zip(widths[:-1], widths[1:]))
    channels = len(_ORDERS[_BASE.get(family, family)])
    point = widths[0] + (n_res if family in ("helmholtz", "burgers_loss", "cavity_loss") else 0)
    if not case["call"].startswith("train"):
        point += n_res
    copies = {"forward": 1, "backward": 2}.get(case["call"], 6)  # params; params, grad; params, m, v in and out
    gemm = 2.0 * channels * sum(a * b for a, b in zip(widths[1:-1], widths[2:]))
    return {"bytes": elem * (n * point + copies * n_par) + 8,
            "flops": n * gemm * (1 if case["call"] == "forward" else 3)}


# ------------------------------------------------------------------ float64 values
def _partitions(items):
    if not items:
        yield []
        return
    for part in _partitions(items[1:]):
        yield [[items[0]]] + part
        for i in range(len(part)):
            yield part[:i] + [[items[0]] + part[i]] + part[i + 1:]


def _tanh_jet(z):
    """Derivative channels of tanh(z) from those of z: the sum over set partitions of each channel's letters."""
    a = torch.tanh(z[""])
    s = 1.0 - a * a
    phi = [a, s, -2.0 * a * s, s * (6.0 * a * a - 2.0), 8.0 * a * s * (2.0 - 3.0 * a * a)]
    out = {}
    for al in z:
        terms = {}
        for part in _partitions(list(al)):
            key = tuple(sorted("".join(sorted(b)) for b in part))
            terms[key] = terms.get(key, 0) + 1
        total = 0.0
        for key, count in terms.items():
            prod = count * phi[len(key)]
            for b in key:
                prod = prod * z[b]
            total = total + prod
        out[al] = total
    return out


def _jets(family, layers, X):
    """Output channels {letters: [n, n_out]}."""
    axes = _AXES[family]
    chans = ["".join(sorted(c)) for c in _ORDERS[family]]
    W, b = layers[0]
    zero = torch.zeros(X.shape[0], W.shape[0], dtype=X.dtype, device=X.device)
    z = {c: X @ W.T + b if c == "" else zero + W[:, axes.index(c)] if len(c) == 1 else zero for c in chans}
    for W, b in layers[1:]:
        a = _tanh_jet(z)
        z = {c: a[c] @ W.T + (b if c == "" else 0.0) for c in chans}
    return z


def _residual(family, coefs, u, src):
    """Residual components [n, n_res]."""
    if family in ("burgers", "allen_cahn", "ks", "helmholtz"):
        u = {c: x[:, 0] for c, x in u.items()}
    if family == "burgers":
        r = [u["t"] + u[""] * u["x"] - coefs["nu"] * u["xx"]]
    elif family == "allen_cahn":
        r = [u["t"] - coefs["eps"] * u["xx"] + coefs["k"] * (u[""] ** 3 - u[""])]
    elif family == "ks":
        r = [u["t"] + coefs["c1"] * u[""] * u["x"] + coefs["c2"] * u["xx"] + coefs["c4"] * u["xxxx"]]
    elif family == "helmholtz":
        r = [u["xx"] + u["yy"] + u["zz"] + coefs["k"] ** 2 * u[""] - src[:, 0]]
    elif family == "ns_uvp":
        U, V = ({c: x[:, o] for c, x in u.items()} for o in (0, 1))
        r = [U["x"] + V["y"]]
        for q, dp in ((U, u["x"][:, 2]), (V, u["y"][:, 2])):
            r.append(U[""] * q["x"] + V[""] * q["y"] + dp - (q["xx"] + q["yy"]) / coefs["Re"])
    else:
        s, nu = {c: x[:, 0] for c, x in u.items()}, coefs["nu"]
        r = [s["ty"] + s["y"] * s["xy"] - s["x"] * s["yy"] + u["x"][:, 1] - nu * (s["xxy"] + s["yyy"]),
             -s["tx"] - s["y"] * s["xx"] + s["x"] * s["xy"] + u["y"][:, 1] + nu * (s["xxx"] + s["xyy"])]
    return torch.stack(r, 1)


def _loss_rows(case, u, X, src):
    """(residual rows [n, n_res], sum of the weighted means' squares) of a composite loss on all its points."""
    a, b, c = _loss_counts(case)
    if case["family"] == "burgers_loss":
        rows = torch.zeros(X.shape[0], 2, dtype=X.dtype, device=X.device)
        bc = torch.cat([u[""], u["x"]], 1)
        bc = bc[0:a:2] - bc[1:a:2]
        ic = u[""][a:a + b] - src[a:a + b, :1]
        pde = _residual("burgers", dict(nu=0.01), {k: x[a + b:] for k, x in u.items()}, None)
        rows[0:a:2], rows[a:a + b, :1], rows[a + b:, :1] = bc.detach(), ic.detach(), pde.detach()
        return rows, bc.square().sum() / (a // 2) + ic.square().sum() / b + pde.square().sum() / c
    rows = torch.zeros(X.shape[0], 3, dtype=X.dtype, device=X.device)
    pde = _residual("ns_uvp", dict(Re=100.0), {k: x[:a] for k, x in u.items()}, None)
    vel = u[""][a:, :2] - src[a:, :2]
    rows[:a], rows[a:, :2] = pde.detach(), vel.detach()
    return rows, pde.square().sum() / a + vel[:b].square().sum() / b + vel[b:].square().sum() / c


def _evaluate(case, ins, want_grad):
    """(residual rows, loss, packed gradient or None) in float64."""
    family = _BASE.get(case["family"], case["family"])
    theta = ins["params"].double().requires_grad_(want_grad)
    widths, layers, off = _network(case), [], 0
    for fi, fo in zip(widths[:-1], widths[1:]):
        layers.append((theta[off:off + fo * fi].view(fo, fi), theta[off + fo * fi:off + fo * fi + fo]))
        off += fo * fi + fo
    X, src = ins["X"].double(), None if ins["source"] is None else ins["source"].double()
    if case["kind"] == "loss":
        chunk = X.shape[0]
    else:
        chunk = max(1024, int(4e9 / (8 * 12 * len(_ORDERS[family]) * case["width"] * case["hidden"])))
    rows, loss, grad = [], 0.0, torch.zeros_like(theta)
    for i in range(0, X.shape[0], chunk):
        x, f = X[i:i + chunk], None if src is None else src[i:i + chunk]
        with torch.set_grad_enabled(want_grad):
            u = _jets(family, layers, x)
            if case["kind"] == "loss":
                r, part = _loss_rows(case, u, x, f)
            else:
                r = _residual(family, case.get("coefs", FAMILIES[family]["coefs"]), u, f)
                part = r.square().sum() / X.shape[0]
        if want_grad:
            grad += torch.autograd.grad(part, theta, retain_graph=True)[0]
        rows.append(r.detach())
        loss = loss + part.detach()
    return torch.cat(rows), loss, grad


def _adam(ins, grad, t):
    """Parameters and moments after Adam step t (beta 0.9 and 0.999, eps 1e-8, bias-corrected)."""
    m = 0.9 * ins["m"].double() + 0.1 * grad
    v = 0.999 * ins["v"].double() + 0.001 * grad * grad
    step = LR * (m / (1.0 - 0.9 ** t)) / ((v / (1.0 - 0.999 ** t)).sqrt() + 1e-8)
    return ins["params"].double() - step, m, v


def exact(case, seed):
    if work(case)["flops"] > 8e12:
        return None  # longer than 20 s in float64 on one GPU
    g = _generator(seed)
    members = _members(case) if case["kind"] == "batch" else [case]
    ins = [_inputs(c, g) for c in members]
    got = [_evaluate(c, x, case["call"] != "forward") for c, x in zip(members, ins)]
    loss = torch.stack([torch.as_tensor(x[1]) for x in got]) if case["kind"] == "batch" else got[0][1]
    if case["call"].startswith("train"):
        new = [_adam(x, y[2], STEP0 + 1) for x, y in zip(ins, got)]
        return {"loss": loss, **{k: torch.cat([x[i] for x in new]) for i, k in enumerate(("params", "m", "v"))}}
    out = {"loss": loss}
    if case["kind"] != "batch":
        out["r"] = got[0][0]
    if case["call"] == "backward":
        out["grad"] = [x[2] for x in got] if case["kind"] == "batch" else got[0][2]
    return out
