"""What is timed: the work that users of the library have it do, through its
public entry points (the C ABI's binding and the autograd wrapper).

A case is a dict of plain values; ``kind`` names the entry point:

* ``net``      one network on its handle, mlp_train_epochs: the fused FP32
               kernel, the bf16 tensor-core kernel or the general kernels,
               whichever the library picks for the shape and precision;
* ``nets``     many independent networks in one launch, mlp_batch_run;
* ``score``    outputs of a trained network on new rows, mlp_forward;
* ``autograd`` forward and backward of the torch function;
* ``zscore``   normalisation of a feature table into the training layout.

Training continues from the state's weights on every pass, as a program that
trains in rounds does.  Loss histories are handed back as float32: they are
sums of FP32 errors.
"""
import math

import numpy as np
import torch

from paper_1908_07847_gb300 import binding as B
from paper_1908_07847_gb300.autograd import mlp

LR = 0.1
PRECS = {"fp32": B.MLP_FP32, "bf16": B.MLP_BF16, "fp64": B.MLP_FP64}
XTYPE = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp64": torch.float64}
ACTS = {"sigmoid": B.MLP_ACT_SIGMOID, "tanh": B.MLP_ACT_TANH}


def listed():
    return [
        # The paper's own size: the 33-marker cohort, 96 training rows, one
        # hidden layer of 16, 1000 epochs a call (progress is looked at every
        # 1000 epochs).  One block holds all rows.
        dict(name="cohort-1000-epochs", kind="net", prec="fp32", act="sigmoid", D=33, H=16, n=96, epochs=1000, mb=0,
             rows_per_block=96),
        # One full-batch epoch of a mid-sized table, the smallest call: a
        # program that steers training epoch by epoch.
        dict(name="step-4096-rows", kind="net", prec="fp32", act="sigmoid", D=33, H=64, n=4096, epochs=1, mb=0),
        # Mini-batch training, ragged everywhere, tanh hidden units.
        dict(name="minibatch-fp32", kind="net", prec="fp32", act="tanh", D=33, H=100, n=20011, epochs=2, mb=1000),
        # The two sex-split subsets trained as separate networks in one launch
        # (the accuracy curves' workload), the plan's default kernel shape.
        dict(name="two-subsets-1000-epochs", kind="nets", prec="fp32", act="sigmoid", D=33, nets=2, H_lo=16, H_hi=16,
             n_lo=44, n_hi=46, epochs=1000, mix=1, shape=0),
        # The benchmark's default line: thousands of small networks of mixed
        # widths and row counts, FP32, the autotuner's kernel shape.
        dict(name="nets-fp32-4096", kind="nets", prec="fp32", act="sigmoid", D=33, nets=4096, H_lo=4, H_hi=128,
             n_lo=50, n_hi=120, epochs=500, mix=2, shape=5),
        # Many larger networks on bf16 rows (33 markers padded to 48).
        dict(name="nets-bf16-1024", kind="nets", prec="bf16", act="sigmoid", D=48, real=33, nets=1024, H_lo=256,
             H_hi=256, n_lo=4096, n_hi=16384, epochs=8, mix=4, shape=-1),
        # One wide network, a million bf16 rows, one epoch of mini-batches.
        dict(name="wide-bf16-1M", kind="net", prec="bf16", act="sigmoid", D=48, real=33, H=2048, n=1 << 20, epochs=1,
             mb=8192),
        # Scoring new rows with the wide network.
        dict(name="score-wide-bf16", kind="score", prec="bf16", act="sigmoid", D=48, real=33, H=2048, n=200003),
        # FP32 training of a network too wide for the fused kernel.
        dict(name="general-fp32", kind="net", prec="fp32", act="sigmoid", D=64, H=512, n=20011, epochs=2, mb=4096),
        # A step of a torch program: outputs, then every weight gradient.
        dict(name="autograd-fp32", kind="autograd", prec="fp32", act="sigmoid", D=33, H=512, n=100003, gX=False),
        # Double precision with the input gradient, as gradient checks and
        # sensitivity studies use it.
        dict(name="autograd-fp64", kind="autograd", prec="fp64", act="tanh", D=33, H=64, n=4096, gX=True),
        # The whole feature table normalised into the padded bf16 layout.
        dict(name="zscore-4M", kind="zscore", D=33, D_out=48, n=4000037, out="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    act = rng.choice(["sigmoid", "sigmoid", "tanh"])
    what = rng.choice(["fused", "minibatch", "nets-fp32", "nets-bf16", "wide", "score", "general", "autograd", "zscore"])
    if what == "fused":
        D, H, n = rng.randint(5, 64), _log_int(rng, 4, 128), _log_int(rng, 40, 20000)
        return dict(kind="net", prec="fp32", act=act, D=D, H=H, n=n, epochs=_log_int(rng, 1, max(1, 200000 // n)), mb=0)
    if what == "minibatch":
        n = _log_int(rng, 1000, 50000)
        mb = _log_int(rng, max(16, n // 500), n)
        return dict(kind="net", prec="fp32", act=act, D=rng.randint(5, 64), H=_log_int(rng, 4, 128), n=n,
                    epochs=rng.randint(1, 3), mb=mb)
    if what == "nets-fp32":
        D = rng.choice([33, 33, rng.randint(5, 36), rng.randint(5, 64)])
        nets, n_hi, H_hi = _log_int(rng, 2, 4096), _log_int(rng, 40, 400), _log_int(rng, 8, 128)
        row_epochs = 2e8 * 33 * 66 / (D * (H_hi + 4) / 2 * nets * n_hi)
        return dict(kind="nets", prec="fp32", act=act, D=D, nets=nets, H_lo=4, H_hi=H_hi, n_lo=n_hi // 2, n_hi=n_hi,
                    epochs=_log_int(rng, 1, max(1, min(500, int(row_epochs)))), mix=rng.randint(0, 1 << 20),
                    shape=rng.choice([0, 5]) if D <= 36 else 0)
    if what == "nets-bf16":
        H = rng.choice([128, 256])
        nets, n_hi = _log_int(rng, 8, 1024), _log_int(rng, 500, 16384)
        D = rng.choice([40, 48, 8 * rng.randint(1, 7)])
        return dict(kind="nets", prec="bf16", act=act, D=D, real=max(1, D - rng.randint(0, 15)), nets=nets, H_lo=H,
                    H_hi=H, n_lo=max(1, n_hi // 4), n_hi=n_hi, epochs=rng.randint(1, 8), mix=rng.randint(0, 1 << 20),
                    shape=-1)
    if what == "wide":
        n, D = _log_int(rng, 3000, 1 << 20), rng.choice([40, 48, 8 * rng.randint(1, 6)])
        return dict(kind="net", prec="bf16", act=act, D=D, real=max(1, D - rng.randint(0, 15)),
                    H=256 * rng.randint(1, 8), n=n, epochs=1, mb=rng.choice([0, _log_int(rng, 1000, 16384)]))
    if what == "score":
        prec = rng.choice(["fp32", "bf16", "bf16", "fp64"])
        D, H = (8 * rng.randint(2, 12), _log_int(rng, 16, 2048)) if prec == "bf16" else (rng.randint(5, 100), _log_int(rng, 16, 1024))
        most = (2e9 if prec != "fp64" else 2e7) / (D * H)
        return dict(kind="score", prec=prec, act=act, D=D, H=H, n=_log_int(rng, 100, max(200, min(1e6, most * 10))))
    if what == "general":
        prec = rng.choice(["fp32", "fp32", "bf16", "fp64"])
        D, H = rng.randint(5, 200), rng.randint(129, 1000)
        n = _log_int(rng, 500, 30000 if prec != "fp64" else 3000)
        return dict(kind="net", prec=prec, act=act, D=D, H=H, n=n, epochs=rng.randint(1, 3),
                    mb=rng.choice([0, _log_int(rng, max(100, n // 20), n)]))
    if what == "autograd":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        D, H = rng.randint(5, 100), _log_int(rng, 8, 1000)
        most = (2e9 if prec == "fp32" else 2e7) / (D * H)
        return dict(kind="autograd", prec=prec, act=act, D=D, H=H, n=_log_int(rng, 50, max(100, min(2e5, most))),
                    gX=rng.random() < 0.5)
    D = rng.choice([33, rng.randint(5, 64), _log_int(rng, 5, 300)])
    out = rng.choice(["bf16", "fp32"])
    return dict(kind="zscore", D=D, D_out=D if out == "fp32" else 8 * ((D + 7) // 8), n=_log_int(rng, 100, 1.2e8 / D),
                out=out)


# --------------------------------------------------------------------- inputs


def _sizes(case):
    """Widths and row counts of a many-nets case (part of the case: work and
    outputs of every seed have the same shapes)."""
    g = np.random.default_rng(case["mix"])
    return (g.integers(case["H_lo"], case["H_hi"], size=case["nets"], endpoint=True),
            g.integers(case["n_lo"], case["n_hi"], size=case["nets"], endpoint=True))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _rows(g, n, D, real, dtype):
    """Standardised features, the padding columns zero, and labels decided by
    a random direction."""
    X = torch.zeros((n, D), dtype=dtype, device="cuda")
    X[:, :real] = torch.randn((n, real), generator=g, device="cuda").to(dtype)
    t = torch.randn(real, generator=g, device="cuda")
    y = (X[:, :real].float() @ t > 0).float()
    return X, y


def _weights(g, D, H, real, dtype):
    """W1 ~ U(+-1/sqrt(D)), w2 ~ U(+-1/sqrt(H)), zero biases and padding."""
    W1 = torch.zeros((H, D), dtype=dtype, device="cuda")
    W1[:, :real] = ((2 * torch.rand((H, real), generator=g, device="cuda") - 1) / math.sqrt(real)).to(dtype)
    w2 = ((2 * torch.rand(H, generator=g, device="cuda") - 1) / math.sqrt(H)).to(dtype)
    z = torch.zeros(H, dtype=dtype, device="cuda")
    return W1, z, w2, torch.zeros(1, dtype=dtype, device="cuda")


def _net_inputs(case, seed):
    g = _gen(seed)
    D, H, n, real, prec = case["D"], case["H"], case["n"], case.get("real", case["D"]), case["prec"]
    wt = torch.float64 if prec == "fp64" else torch.float32
    X, y = _rows(g, n, D, real, XTYPE[prec])
    return X, y.to(wt), _weights(g, D, H, real, wt)


def _nets_inputs(case, seed):
    g = _gen(seed)
    D, real = case["D"], case.get("real", case["D"])
    Hs, ns = _sizes(case)
    X, y = _rows(g, int(ns.sum()), D, real, XTYPE[case["prec"]])
    Hm = int(Hs.max())
    sc = torch.from_numpy(1.0 / np.sqrt(Hs)).to("cuda", torch.float32)
    W1 = torch.zeros((len(Hs), Hm, D), device="cuda")
    W1[:, :, :real] = (2 * torch.rand((len(Hs), Hm, real), generator=g, device="cuda") - 1) / math.sqrt(real)
    w2 = (2 * torch.rand((len(Hs), Hm), generator=g, device="cuda") - 1) * sc[:, None]
    parts = []
    for t, H in enumerate(Hs.tolist()):
        parts += [W1[t, :H].reshape(-1), torch.zeros(H, device="cuda"), w2[t, :H], torch.zeros(1, device="cuda")]
    return X, y, torch.cat(parts), Hs, ns


def _table(case, seed):
    """Raw measurements: every column with its own mean and spread."""
    g = _gen(seed)
    D, n = case["D"], case["n"]
    mean = 200 * torch.rand(D, generator=g, device="cuda") - 20
    sd = torch.exp(4 * torch.rand(D, generator=g, device="cuda") - 1)
    return torch.randn((n, D), generator=g, device="cuda").mul_(sd).add_(mean)


# ------------------------------------------------------------ states and runs


class _Handle:
    """Owns a library handle or plan."""

    def __init__(self, value, free):
        self.value, self.free = value, free

    def __del__(self):
        self.free(self.value)


class _DeviceArray:
    """The handle's packed weights as a device array (keeps the handle)."""

    def __init__(self, handle, count, typestr):
        self.handle = handle
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": typestr, "strides": None, "version": 2,
                                         "data": (B.mlp_weights_device(handle.value), False)}


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _handle(case, W):
    h = _Handle(B.mlp_create(case["D"], case["H"], LR, 1, PRECS[case["prec"]], ACTS[case["act"]]), B.mlp_destroy)
    B.mlp_set_weights(h.value, *[w.cpu().numpy() for w in W])
    return h


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("net", "score"):
        s["X"], s["y"], W = _net_inputs(case, seed)
        s["h"] = _handle(case, W)
        if kind == "net":
            if case.get("rows_per_block"):
                B.mlp_set_rows_per_block(s["h"].value, case["rows_per_block"])
            P = (case["D"] + 2) * case["H"] + 1
            s["w"] = torch.as_tensor(_DeviceArray(s["h"], P, "<f8" if case["prec"] == "fp64" else "<f4"), device="cuda")
            s["loss"] = torch.zeros(case["epochs"], dtype=torch.float64, device="cuda")
        else:
            s["o"] = torch.empty(case["n"], dtype=s["y"].dtype, device="cuda")
    elif kind == "nets":
        X, y, P, Hs, ns = _nets_inputs(case, seed)
        D = case["D"]
        L = torch.zeros((len(Hs), case["epochs"]), dtype=torch.float64, device="cuda")
        r = np.concatenate([[0], np.cumsum(ns)]).tolist()
        p = np.concatenate([[0], np.cumsum((D + 2) * Hs + 1)]).tolist()
        descs = [B.mlp_net_desc(int(Hs[t]), int(ns[t]), X.data_ptr() + r[t] * D * X.element_size(),
                                y.data_ptr() + 4 * r[t], P.data_ptr() + 4 * p[t], L.data_ptr() + 8 * case["epochs"] * t)
                 for t in range(len(Hs))]
        plan = _Handle(B.mlp_batch_create(PRECS[case["prec"]], ACTS[case["act"]], D, descs, LR, 1), B.mlp_batch_destroy)
        if case["shape"] > 0:
            B.mlp_batch_set_shape(plan.value, case["shape"])
        s.update(X=X, y=y, P=P, L=L, plan=plan)
    elif kind == "autograd":
        s["X"], _, W = _net_inputs(case, seed)
        s["X"].requires_grad_(case["gX"])
        s["W"] = [w.requires_grad_(True) for w in W]
        s["go"] = torch.randn(case["n"], generator=_gen(seed + 1), device="cuda", dtype=s["X"].dtype)
    else:
        D = case["D"]
        s["X"] = _table(case, seed)
        s["Y"] = torch.empty((case["n"], case["D_out"]), dtype=XTYPE[case["out"]], device="cuda")
        s["mean"] = torch.empty(D, dtype=torch.float64, device="cuda")
        s["sdev"] = torch.empty(D, dtype=torch.float64, device="cuda")
        s["bytes"] = B.mlp_zscore_workspace_bytes(D)
        s["ws"] = torch.empty(s["bytes"], dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "net":
        B.mlp_train_epochs(s["h"].value, s["X"], s["y"], case["n"], case["epochs"], case["mb"], s["loss"], None, _stream())
        return [s["w"], s["loss"].float()]
    if kind == "nets":
        B.mlp_batch_run(s["plan"].value, case["epochs"], _stream())
        return [s["P"], s["L"].float()]
    if kind == "score":
        B.mlp_forward(s["h"].value, s["X"], case["n"], s["o"], _stream())
        return s["o"]
    if kind == "autograd":
        o = mlp(s["X"], *s["W"], ACTS[case["act"]])
        wrt = ([s["X"]] if case["gX"] else []) + s["W"]
        return [o.detach(), *torch.autograd.grad(o, wrt, s["go"])]
    B.mlp_zscore(s["X"], case["n"], case["D"], _n_fit(case), PRECS[case["out"]], case["D_out"], s["Y"], s["mean"],
                 s["sdev"], s["ws"], s["bytes"], _stream())
    return [s["Y"], s["mean"], s["sdev"]]


def _n_fit(case):
    return max(1, (3 * case["n"]) // 4)   # the training split


# ----------------------------------------------------------------------- work


def work(case):
    kind = case["kind"]
    if kind == "zscore":
        n, D = case["n"], case["D"]
        return {"bytes": n * (4 * D + (2 if case["out"] == "bf16" else 4) * case["D_out"]) + 16 * D,
                "flops": 3 * n * D + 4 * _n_fit(case) * D}
    D = case["D"]
    e = {"fp32": 4, "bf16": 2, "fp64": 8}[case["prec"]]
    w = 8 if case["prec"] == "fp64" else 4
    if kind == "nets":
        Hs, ns = _sizes(case)
        ep = case["epochs"]
        return {"bytes": int(ns.sum()) * (D * e + 4) + 8 * int(((D + 2) * Hs + 1).sum()) + 8 * ep * case["nets"],
                "flops": float((ns * Hs).sum()) * (4 * D + 10) * ep}
    H, n = case["H"], case["n"]
    P = (D + 2) * H + 1
    if kind == "net":
        return {"bytes": n * (D * e + w) + 2 * w * P + 8 * case["epochs"], "flops": n * H * (4.0 * D + 10) * case["epochs"]}
    if kind == "score":
        return {"bytes": n * (D * e + w) + w * P, "flops": n * H * (2.0 * D + 3)}
    return {"bytes": n * (D * e * (2 if case["gX"] else 1) + 2 * w) + 2 * w * P,
            "flops": n * H * ((6.0 if case["gX"] else 4.0) * D + 10)}


# ------------------------------------------------- the same numbers in 64 bits


def _f(z, act):
    return torch.tanh(z) if act == "tanh" else torch.sigmoid(z)


def _df(h, act):
    return 1 - h * h if act == "tanh" else h * (1 - h)


def _train64(X, y, W1, b1, w2, b2, ns, live, act, epochs, mb):
    """Gradient descent of a batch of networks in 64 bits: X [B, n, D], y and
    the row mask from ns [B], W1 [B, H, D], live [B, H] marks real units.
    Returns the weights and the loss histories [B, epochs]."""
    lr = float(np.float32(LR))
    n = X.shape[1]
    mb = n if mb <= 0 or mb >= n else mb
    hist = torch.zeros((X.shape[0], epochs), dtype=torch.float64, device=X.device)
    rows = torch.arange(n, device=X.device)[None, :] < ns[:, None]
    for e in range(epochs):
        for r in range(0, n, mb):
            Xb, yb, on = X[:, r:r + mb], y[:, r:r + mb], rows[:, r:r + mb]
            c = 1.0 / on.sum(1, keepdim=True)
            h = _f(torch.baddbmm(b1[:, None, :], Xb, W1.transpose(1, 2)), act)
            o = torch.sigmoid(torch.bmm(h, w2[:, :, None])[:, :, 0] + b2)
            err = torch.where(on, o - yb, 0.0)
            hist[:, e] += 0.5 * (err * err).sum(1) / ns
            d2 = c * err * o * (1 - o)
            d1 = d2[:, :, None] * w2[:, None, :] * _df(h, act)
            gw2 = torch.bmm(d2[:, None, :], h)[:, 0] * live
            W1 = torch.baddbmm(W1, d1.transpose(1, 2), Xb, alpha=-lr)
            b1, w2, b2 = b1 - lr * d1.sum(1), w2 - lr * gw2, b2 - lr * d2.sum(1, keepdim=True)
    return W1, b1, w2, b2, hist


def exact(case, seed):
    if work(case)["flops"] > 1.2e13:
        return None
    kind = case["kind"]
    if kind == "zscore":
        X = _table(case, seed).double()
        fit = X[:_n_fit(case)]
        mean = fit.mean(0)
        sdev = (fit - mean).square().mean(0).sqrt()
        Y = torch.zeros((case["n"], case["D_out"]), dtype=torch.float64, device="cuda")
        Y[:, :case["D"]] = torch.where(sdev > 0, (X - mean) / torch.where(sdev > 0, sdev, 1.0), 0.0)
        return [Y, mean, sdev]
    act = case["act"]
    if kind == "nets":
        X, y, P, Hs, ns = _nets_inputs(case, seed)
        D, ep = case["D"], case["epochs"]
        r = np.concatenate([[0], np.cumsum(ns)])
        p = np.concatenate([[0], np.cumsum((D + 2) * Hs + 1)])
        out, hist = P.double(), torch.zeros((len(Hs), ep), dtype=torch.float64, device="cuda")
        # nets of similar row counts side by side, up to about 1 GB an activation
        order = np.argsort(ns, kind="stable")
        step = max(1, int(1.2e8 / (int(ns.max()) * int(Hs.max()))))
        for c0 in range(0, len(order), step):
            ids = order[c0:c0 + step]
            b, nm, Hm = len(ids), int(ns[ids].max()), int(Hs[ids].max())
            z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
            Xb, yb, W1, b1, w2, b2, live = z(b, nm, D), z(b, nm), z(b, Hm, D), z(b, Hm), z(b, Hm), z(b, 1), z(b, Hm)
            for i, t in enumerate(ids):
                H, HD, q = int(Hs[t]), int(Hs[t]) * D, P[int(p[t]):int(p[t + 1])].double()
                Xb[i, :ns[t]], yb[i, :ns[t]] = X[r[t]:r[t + 1]].double(), y[r[t]:r[t + 1]].double()
                W1[i, :H], b1[i, :H], w2[i, :H], b2[i] = q[:HD].view(H, D), q[HD:HD + H], q[HD + H:HD + 2 * H], q[-1]
                live[i, :H] = 1
            W1, b1, w2, b2, hs = _train64(Xb, yb, W1, b1, w2, b2, torch.from_numpy(ns[ids]).cuda(), live, act, ep, 0)
            for i, t in enumerate(ids):
                H = int(Hs[t])
                out[int(p[t]):int(p[t + 1])] = torch.cat([W1[i, :H].reshape(-1), b1[i, :H], w2[i, :H], b2[i]])
                hist[t] = hs[i]
        return [out, hist]
    X, y, W = _net_inputs(case, seed)
    W1, b1, w2, b2 = [w.double() for w in W]
    X = X.double()
    if kind == "net":
        n, H = case["n"], case["H"]
        live = torch.ones((1, H), dtype=torch.float64, device="cuda")
        W1, b1, w2, b2, hist = _train64(X[None], y.double()[None], W1[None], b1[None], w2[None], b2[None],
                                        torch.tensor([n], device="cuda"), live, act, case["epochs"], case["mb"])
        return [torch.cat([W1.reshape(-1), b1.reshape(-1), w2.reshape(-1), b2.reshape(-1)]), hist[0]]
    if kind == "score":
        step = max(1, int(1.2e8 / case["H"]))
        return torch.cat([torch.sigmoid(_f(X[r:r + step] @ W1.T + b1, act) @ w2 + b2) for r in range(0, len(X), step)])
    go = torch.randn(case["n"], generator=_gen(seed + 1), device="cuda", dtype=XTYPE[case["prec"]]).double()
    h = _f(X @ W1.T + b1, act)
    o = torch.sigmoid(h @ w2 + b2)
    d2 = go * o * (1 - o)
    d1 = d2[:, None] * w2 * _df(h, act)
    return [o] + ([d1 @ W1] if case["gX"] else []) + [d1.T @ X, d1.sum(0), h.T @ d2, d2.sum().reshape(1)]
