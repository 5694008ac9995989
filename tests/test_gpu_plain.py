"""The general kernels (any D and H) at the edges of their tiles: row tiles of
16 to 128 rows picked by the grid's size, inputs staged in slices of up to 64,
gradient tiles of 64 inputs in quads with 2 to 32 row subsets, input-gradient
row groups; forward, upstream-gradient backward and a training step against the
oracle at the FP32 bars (1e-12 in FP64)."""
import numpy as np
import pytest

import oracle
from oracle import Params
from paper_1908_07847_gb300 import binding as B
from tests.gpu_util import FWD_TOL, GRAD_TOL, W_TOL, Net, dev, host, lr32, problem, rel_err_elem, rel_err_norm, stream

pytestmark = pytest.mark.gpu

#        rows, D, H: one row; slices 65 = 33 + 32; 128-row tiles; 64-row tiles; two
#        input tiles; three; one quad; quads of 2 inputs with 16 subsets; aligned hid
SHAPES = [(1, 1, 1), (33, 65, 65), (40001, 36, 70), (20003, 33, 64), (2500, 65, 300), (77, 130, 67), (513, 3, 129),
          (1025, 7, 31), (4096, 64, 512), (17, 64, 130), (15, 49, 200)]


@pytest.mark.parametrize("n,D,H", SHAPES)
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_forward_and_upstream_gradients(n, D, H, dtype):
    import torch
    from paper_1908_07847_gb300.autograd import mlp
    if dtype == "float64" and n * D * H > 4e7:
        n = 3001
    act = (n + H) % 2
    X, _, W = problem(7000 + n + H, n, D, H)
    dt = getattr(torch, dtype)
    rng = np.random.default_rng(n)
    go = rng.normal(size=n).astype(np.float32)
    t = [dev(np.asarray(a, np.float32)).to(dt).requires_grad_(True) for a in (X, *W)]
    o = mlp(*t, act)
    g = torch.autograd.grad(o, t, dev(go).to(dt))
    p = Params(*[np.asarray(a, np.float64) for a in W])
    _, o_ref = oracle.forward(X, p, act)
    gW1, gb1, gw2, gb2, gX = oracle.backward(X, p, go.astype(np.float64), act, want_gX=True)
    ft, gt = (FWD_TOL, GRAD_TOL) if dtype == "float32" else (1e-12, 1e-12)
    assert rel_err_elem(host(o), o_ref) <= ft
    for got, want in zip(g, (gX, gW1, gb1, gw2, gb2)):
        assert rel_err_norm(host(got), want) <= gt


@pytest.mark.parametrize("n,D,H,mb", [(300, 70, 129, 0), (1000, 33, 300, 260), (65, 64, 513, 64)])
@pytest.mark.parametrize("loss_mean", [0, 1])
def test_training_steps_update_and_loss(n, D, H, mb, loss_mean):
    """Gradient reduction, update and loss in one kernel: weights, loss and
    gradient-norm histories of three epochs against the oracle."""
    import torch
    X, y, W = problem(7100 + n, n, D, H)
    lr = 0.1 if loss_mean else 0.1 / n
    lh = torch.zeros(3, dtype=torch.float64, device="cuda")
    gh = torch.zeros(3, dtype=torch.float64, device="cuda")
    with Net(D, H, lr=lr, loss_mean=loss_mean) as net:
        net.set(W)
        B.mlp_train_epochs(net.h, dev(X), dev(y), n, 3, mb, lh, gh, stream())
        assert net.check() == B.MLP_OK
        got = net.flat()
    q, l_ref, g_ref = oracle.train(X, y, Params(*W), lr32(lr), 3, minibatch=mb, loss_mean=bool(loss_mean))
    assert rel_err_norm(got, q.flat()) <= W_TOL
    np.testing.assert_allclose(host(lh), l_ref, rtol=1e-6)
    np.testing.assert_allclose(host(gh), g_ref, rtol=1e-4)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("n,D,H", [(16300, 12, 65), (32700, 33, 68), (16300, 47, 127), (21001, 48, 200), (2433, 64, 772),
                                   (20001, 16, 129), (300, 49, 7296), (33001, 40, 128)])
def test_tensor_core_forward(n, D, H, prec):
    """The split forward (12 to 64 inputs, H > 64, at least 128 tiles; with hid
    more than 32 inputs, H % 4 = 0 and at least 8192 inputs x tiles): every K step,
    remainders of rows and units, hid with and without 16-byte rows, at the
    FP32 bar; hidden activations within the bound of an FP32 sum of D + 1 terms,
    (D + 1) 2^-24 sum |x w|, and 1e-6 of their value for the activation (its
    slope is at most 1)."""
    import torch
    from paper_1908_07847_gb300 import inputs as I
    act = D % 2
    X, _, W = problem(7300 + n + D, n, D, H)
    if prec == "bf16":
        X = I.bf16_round(X)
    with Net(D, H, prec=B.MLP_BF16 if prec == "bf16" else B.MLP_FP32, act=act) as net:
        net.set(W)
        o = torch.zeros(n, device="cuda")
        B.mlp_forward(net.h, dev(X).to(torch.bfloat16 if prec == "bf16" else torch.float32), n, o, stream())
        plain, hid = host(o), None
    if prec == "fp32":
        t = [dev(np.asarray(a, np.float32)) for a in (X, *W)]
        hd, o = torch.zeros((n, H), device="cuda"), torch.zeros(n, device="cuda")
        nb = B.mlp_workspace_bytes(B.MLP_FP32, D, H, n)
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        B.mlp_forward_w(B.MLP_FP32, act, D, H, n, *t, hd, o, ws, nb, stream())
        got, hid = host(o), host(hd)
    h_ref, o_ref = oracle.forward(X, Params(*W), act)
    assert rel_err_elem(plain, o_ref) <= FWD_TOL
    if hid is not None:
        assert rel_err_elem(got, o_ref) <= FWD_TOL
        size = np.abs(X.astype(np.float64)) @ np.abs(W[0].astype(np.float64)).T + np.abs(W[1])
        assert np.all(np.abs(hid - h_ref) <= (D + 1) * 2.0 ** -24 * size + 1e-6 * np.abs(h_ref))


@pytest.mark.parametrize("where", ["x", "w"])
def test_tensor_core_forward_of_values_outside_the_parts_range(where):
    """Infinities, NaN, huge and tiny values in one row (or one unit's
    weights): those tiles take plain FP32 multiply-adds, the others do not
    notice.  An infinite input saturates its units as in 64 bits."""
    import torch
    n, D, H = 8400, 33, 130
    X, _, W = problem(7400, n, D, H)
    X[7, 3], X[200, 0], X[333, 1], X[500, 2], X[600, 5] = np.inf, -np.inf, 3.3e38, 1e-38, np.nan
    if where == "w":
        W[0][5, 4], W[0][129, 0] = 1e30, 1e-35
    with Net(D, H) as net:
        net.set(W)
        o = torch.zeros(n, device="cuda")
        B.mlp_forward(net.h, dev(X), n, o, stream())
        got = host(o)
    with np.errstate(all="ignore"):
        _, ref = oracle.forward(X, Params(*W))
    assert np.isnan(got[600]) and np.isnan(ref[600])
    ok = np.arange(n) != 600
    assert rel_err_elem(got[ok], ref[ok]) <= FWD_TOL


@pytest.mark.parametrize("prec,D,H,n", [("fp32", 33, 2000, 9000), ("fp32", 12, 1940, 9000), ("fp32", 64, 2048, 8100),
                                        ("bf16", 48, 2000, 14000), ("bf16", 19, 2048, 13000)])
def test_tensor_core_forward_between_plain_tiles(prec, D, H, n):
    """Blocks that walk over several tiles, some outside the parts' range (every
    third tile, by one row) and some not: units go back and forth between their
    parts and their plain form, with remainders of inputs, rows and units, and
    once with a block of units that never has parts (a weight of 1e-33)."""
    import torch
    from paper_1908_07847_gb300 import inputs as I
    X, _, W = problem(7500 + D, n, D, H)
    for r, v in zip(range(5, n, 384), [np.inf, -2.0 ** 62, 3e38, 1e-33] * n):
        X[r, r % D] = v
    if prec == "bf16":
        X = I.bf16_round(X)
    W[0][H - 1, 1] = 1e-33
    with Net(D, H, prec=B.MLP_BF16 if prec == "bf16" else B.MLP_FP32) as net:
        net.set(W)
        o = torch.zeros(n, device="cuda")
        B.mlp_forward(net.h, dev(X).to(torch.bfloat16 if prec == "bf16" else torch.float32), n, o, stream())
        got = host(o)
    with np.errstate(all="ignore"):
        _, ref = oracle.forward(X, Params(*W))
    assert np.all(np.isfinite(ref)) and rel_err_elem(got, ref) <= FWD_TOL


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_plain_tiles_of_the_tensor_core_forward_are_not_slow(prec):
    """A fit that diverged, or one tiny or infinite weight a block of units, sends
    every tile through multiply-adds: some five times the clean call's time, 20 to 90
    times when each multiply-add loaded its operands.  Bound: 10."""
    import torch
    n, D, H = 100003, 48, 1024
    X = torch.randn((n, D), device="cuda").to(torch.bfloat16 if prec == "bf16" else torch.float32)
    o = torch.zeros(n, device="cuda")
    times = []
    for bad in (False, True):
        _, _, W = problem(7600, 16, D, H)
        if bad:
            W[0][::128, 3] = 1e-33
        with Net(D, H, prec=B.MLP_BF16 if prec == "bf16" else B.MLP_FP32) as net:
            net.set(W)
            t = []
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                B.mlp_forward(net.h, X, n, o, stream())
                b.record()
                torch.cuda.synchronize()
                t.append(a.elapsed_time(b))
        times.append(min(t[1:]))
    assert times[1] <= 10 * times[0], times


@pytest.mark.parametrize("D,H,n", [(64, 256, 8192), (48, 260, 16384), (49, 384, 8192)])
def test_tensor_core_forward_of_rows_with_one_dominant_term(D, H, n):
    """Log-normal inputs and weights of one sign: every accumulation of full size
    rounds towards zero, half a unit of the last place on average, 4.3e-8 of the
    sum.  Two accumulators meet two of them at most where the sum lies: the mean
    error of the activations within 1.3e-7 with their own rounding (tanh of values
    below 0.1); four reach 2e-7."""
    import torch
    rng = np.random.default_rng(D)
    X = np.exp(3 * rng.normal(size=(n, D))).astype(np.float32)
    X /= X.sum(1, keepdims=True) * 10
    W = (rng.uniform(size=(H, D)).astype(np.float32), np.zeros(H, np.float32), np.ones(H, np.float32), np.zeros(1, np.float32))
    hd, o = torch.zeros((n, H), device="cuda"), torch.zeros(n, device="cuda")
    nb = B.mlp_workspace_bytes(B.MLP_FP32, D, H, n)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    B.mlp_forward_w(B.MLP_FP32, B.MLP_ACT_TANH, D, H, n, dev(X), *[dev(w) for w in W], hd, o, ws, nb, stream())
    ref = np.tanh(X.astype(np.float64) @ W[0].astype(np.float64).T)
    assert abs(np.mean(host(hd) / ref - 1)) <= 1.3e-7


@pytest.mark.parametrize("prec,D,H", [("fp32", 33, 512), ("bf16", 48, 2048)])
def test_scores_in_pieces_agree_with_scores_at_once(prec, D, H):
    """A table scored at once (tensor cores) and 500 rows at a time (multiply-add
    chains): each within the forward bar of the oracle, so within twice of each
    other; labels differ only where o is that near 0.5.  The same call again gives
    the same bits."""
    import torch
    n = 20000
    X, _, W = problem(7700, n, D, H)
    Xd = dev(X).to(torch.bfloat16 if prec == "bf16" else torch.float32)
    whole, again, pieces = (torch.zeros(n, device="cuda") for _ in range(3))
    lab, labp = (torch.zeros(n, dtype=torch.int8, device="cuda") for _ in range(2))
    with Net(D, H, prec=B.MLP_BF16 if prec == "bf16" else B.MLP_FP32) as net:
        net.set(W)
        B.mlp_forward(net.h, Xd, n, whole, stream())
        B.mlp_forward(net.h, Xd, n, again, stream())
        B.mlp_predict(net.h, Xd, n, lab, stream())
        for i in range(0, n, 500):
            B.mlp_forward(net.h, Xd[i:i + 500], 500, pieces[i:i + 500], stream())
            B.mlp_predict(net.h, Xd[i:i + 500], 500, labp[i:i + 500], stream())
        torch.cuda.synchronize()
    assert torch.equal(whole, again)
    assert rel_err_elem(host(pieces), host(whole)) <= 2 * FWD_TOL
    o = host(whole).astype(np.float64)
    assert np.array_equal(host(lab), (o >= 0.5).astype(np.int8))
    assert np.all(np.abs(o - 0.5)[host(lab) != host(labp)] <= FWD_TOL)


@pytest.mark.parametrize("n,D,H", [(1, 16, 65), (777, 16, 66), (4096, 5, 67), (2500, 16, 385), (9000, 70, 130)])
@pytest.mark.parametrize("act", [0, 1])
def test_fp64_forward_with_a_last_tile_of_few_units(n, D, H, act):
    """One, two and three units in the last tile of 64 (activations that no thread
    needs are skipped there), with and without stored activations."""
    import torch
    X, _, W = problem(7800 + n, n, D, H)
    t = [dev(np.asarray(a, np.float64)) for a in (X, *W)]
    nb = B.mlp_workspace_bytes(B.MLP_FP64, D, H, n)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    h_ref, o_ref = oracle.forward(X, Params(*[np.asarray(a, np.float64) for a in W]), act)
    for store in (False, True):
        hd, o = torch.zeros((n, H), device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.float64)
        B.mlp_forward_w(B.MLP_FP64, act, D, H, n, *t, hd if store else None, o, ws, nb, stream())
        assert rel_err_elem(host(o), o_ref) <= 1e-12
        if store:
            assert rel_err_norm(host(hd), h_ref) <= 1e-12


@pytest.mark.parametrize("D,H,n", [(40, 2000, 9000), (33, 516, 20011), (64, 388, 8300)])
def test_stored_activations_of_plain_tiles(D, H, n):
    """Activations and outputs of tiles outside the parts' range (tiny and huge
    values in some rows, a tiny weight in the last block of units) beside tiles
    within it, with remainders of rows and units: the bound of an FP32 sum of
    D + 1 terms and 1e-6 of their value for the activation."""
    import torch
    X, _, W = problem(7900 + D, n, D, H)
    for r, v in zip(range(9, n, 300), [1e-33, -3e-32, 2.0 ** 61, -1e-36] * n):
        X[r, r % D] = v
    W[0][H - 2, 1] = -1e-33
    t = [dev(np.asarray(a, np.float32)) for a in (X, *W)]
    hd, o = torch.zeros((n, H), device="cuda"), torch.zeros(n, device="cuda")
    nb = B.mlp_workspace_bytes(B.MLP_FP32, D, H, n)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    B.mlp_forward_w(B.MLP_FP32, B.MLP_ACT_SIGMOID, D, H, n, *t, hd, o, ws, nb, stream())
    h_ref, o_ref = oracle.forward(X, Params(*W))
    assert rel_err_elem(host(o), o_ref) <= FWD_TOL
    size = np.abs(X.astype(np.float64)) @ np.abs(W[0].astype(np.float64)).T + np.abs(W[1])
    assert np.all(np.abs(host(hd) - h_ref) <= (D + 1) * 2.0 ** -24 * size + 1e-6 * np.abs(h_ref))
