"""Z-score normalisation on the GPU (Sec. 2.2 normalises the data; read as the
training rows' per-column mean and population deviation) against the oracle:
statistics within 1e-12 relative (FP64 sums in another order), FP32 outputs
within a few float ulps, bf16 outputs within one bf16 ulp; padding exactly 0."""
import numpy as np
import pytest

import oracle
from paper_1908_07847_gb300 import binding as B
from paper_1908_07847_gb300 import inputs as I
from tests.gpu_util import dev, host, stream

pytestmark = pytest.mark.gpu


def table(seed, n, D):
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(n, D)) * rng.uniform(0.2, 5.0, D) + rng.uniform(-50.0, 50.0, D)
    X[:, min(3, D - 1)] = 7.25    # a constant column
    return X.astype(np.float32)


def run(X, n_fit, prec, D_out):
    import torch
    n, D = X.shape
    ws = B.mlp_zscore_workspace_bytes(D)
    W = torch.empty(ws, dtype=torch.uint8, device="cuda")
    Y = torch.full((n, D_out), 99, dtype=torch.float32 if prec == B.MLP_FP32 else torch.int16, device="cuda")
    m = torch.zeros(D, dtype=torch.float64, device="cuda")
    s = torch.zeros(D, dtype=torch.float64, device="cuda")
    B.mlp_zscore(dev(X), n, D, n_fit, prec, D_out, Y, m, s, W, ws, stream())
    torch.cuda.synchronize()
    return host(Y), host(m), host(s)


def bf16_to_float(bits):
    return (bits.astype(np.uint16).astype(np.uint32) << 16).view(np.float32)


@pytest.mark.parametrize("n,D,n_fit", [(1, 5, 1), (100, 33, 75), (1000, 33, 1000), (5000, 33, 3750), (300, 300, 200)])
def test_fp32_output_and_statistics(n, D, n_fit):
    X = table(n + D, n, D)
    Y, m, s = run(X, n_fit, B.MLP_FP32, D)
    Yr, mr, sr = oracle.zscore(X.astype(np.float64), n_fit)
    np.testing.assert_allclose(m, mr, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(s, sr, rtol=1e-12, atol=1e-300)
    # FP32: the two-float mean keeps x - m within a float ulp of |x - m|, the
    # scaling adds one rounding: a few ulps of max(|y|, 1)
    tol = 4 * np.finfo(np.float32).eps * np.maximum(np.abs(Yr), 1.0)
    assert np.all(np.abs(Y - Yr) <= tol)
    assert np.all(Y[:, s == 0.0] == 0.0)


def test_bf16_padded_output_is_the_tensor_core_input():
    """33 columns normalised, converted to bf16 and zero-padded to 48."""
    n, D, n_fit = 65536, 33, I.split_count(65536)
    X = table(7, n, D)
    Yb, m, s = run(X, n_fit, B.MLP_BF16, 48)
    Yr, mr, sr = oracle.zscore(X.astype(np.float64), n_fit)
    got = bf16_to_float(Yb)
    assert np.all(Yb[:, D:] == 0)
    ref = I.bf16_round(Yr.astype(np.float32)).astype(np.float64)
    ulp = np.maximum(np.abs(ref), 2.0 ** -126) * 2.0 ** -7
    assert np.all(np.abs(got[:, :D] - ref) <= ulp)
    assert np.mean(got[:, :D] == ref) > 0.999


def test_deterministic_and_rejects_bad_arguments():
    X = table(3, 2000, 33)
    a = run(X, 1500, B.MLP_FP32, 33)
    b = run(X, 1500, B.MLP_FP32, 33)
    for u, v in zip(a, b):
        assert np.array_equal(u, v)
    import torch
    ws = B.mlp_zscore_workspace_bytes(33)
    W = torch.empty(ws, dtype=torch.uint8, device="cuda")
    Y = torch.empty((10, 33), device="cuda")
    m = torch.empty(33, dtype=torch.float64, device="cuda")
    for n_fit, D_out, wsb in [(0, 33, ws), (11, 33, ws), (5, 32, ws), (5, 33, 8)]:
        with pytest.raises(B.MLPError) as e:
            B.mlp_zscore(dev(X[:10]), 10, 33, n_fit, B.MLP_FP32, D_out, Y, m, m, W, wsb, stream())
        assert e.value.status == B.MLP_EINVAL


@pytest.mark.parametrize("n,D", [(200_003, 33), (120_001, 5), (60_000, 17), (90_001, 300)])
def test_statistics_of_long_tables_and_extreme_columns(n, D):
    """Row counts where a block's rows are added in groups of 16 and 4 with a
    remainder, with columns outside the range of the groups' FP32 sums: huge,
    tiny, constant, offset by 1e7 deviations, infinite and NaN.  Finite columns
    against numpy's 64-bit sums: an FP64 sum of n terms in blocks of a few
    hundred rows is within 1e-12 of it; the mean of a column centred on 0 is
    that much of its deviation, and the deviation of the offset column carries
    the 1e7 of its offset in the mean's rounding only (1e-12 holds)."""
    X = table(11 + D, n, D).astype(np.float64)
    rng = np.random.default_rng(5)
    X[:, 0] = rng.normal(size=n) * 1e30
    X[:, 1] = rng.normal(size=n) * 1e-30
    X[:, 2] = np.float32(1e4) + rng.normal(size=n) * 1e-3
    X[5, D - 1] = np.inf if D > 5 else 1.0
    if D > 5:
        X[n // 2, D - 2] = np.nan
    X = X.astype(np.float32)
    Y, m, s = run(X, n, B.MLP_FP32, D)
    X = X.astype(np.float64)
    ok = np.isfinite(X).all(0)
    mr, sr = X.mean(0), X.std(0)
    assert np.all(np.abs(m - mr)[ok] <= 1e-12 * (np.abs(mr) + sr)[ok])
    np.testing.assert_allclose(s[ok], sr[ok], rtol=1e-12, atol=0)
    assert s[3] == 0.0 and np.all(Y[:, 3] == 0.0)
    if D > 5:
        assert np.isposinf(m[D - 1]) and np.isnan(m[D - 2]) and np.isnan(s[D - 1]) and np.isnan(s[D - 2])


@pytest.mark.parametrize("prec,D,D_out,n", [(B.MLP_FP32, 33, 33, 64), (B.MLP_FP32, 33, 35, 129), (B.MLP_FP32, 3, 3, 7),
                                            (B.MLP_BF16, 33, 37, 65), (B.MLP_BF16, 256, 256, 19), (B.MLP_FP32, 5, 21, 1000),
                                            (B.MLP_BF16, 257, 264, 9), (B.MLP_FP32, 1, 300, 300)])
def test_tiled_and_plain_apply_agree(prec, D, D_out, n):
    """16-byte aligned buffers (tiles) and buffers one element off (an element
    a thread): the same bits for every width, remainder and padding."""
    import torch
    X = dev(table(17 + n, n, D))
    ws = B.mlp_zscore_workspace_bytes(D)
    W = torch.empty(ws, dtype=torch.uint8, device="cuda")
    m = torch.zeros(D, dtype=torch.float64, device="cuda")
    s = torch.zeros(D, dtype=torch.float64, device="cuda")
    dt = torch.int32 if prec == B.MLP_FP32 else torch.int16
    out = []
    for off in (0, 1):
        buf = torch.full((n * D_out + 2,), 99, dtype=dt, device="cuda")
        B.mlp_zscore(X, n, D, n, prec, D_out, buf[off:off + n * D_out], m, s, W, ws, stream())
        out.append(host(buf[off:off + n * D_out]))
        assert int(buf[off + n * D_out]) == 99
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("prec,D,D_out,n", [(B.MLP_FP32, 33, 33, 2000), (B.MLP_FP32, 33, 35, 2129), (B.MLP_FP32, 3, 3, 22007),
                                            (B.MLP_BF16, 33, 37, 2065), (B.MLP_BF16, 256, 256, 275), (B.MLP_FP32, 5, 21, 4001),
                                            (B.MLP_BF16, 257, 264, 300), (B.MLP_FP32, 1, 300, 300), (B.MLP_BF16, 33, 48, 1365),
                                            (B.MLP_BF16, 33, 48, 1366)])
def test_tiled_and_plain_apply_agree_on_tables_that_take_tiles(prec, D, D_out, n):
    """As above for tables beyond 2^16 values, from where aligned outputs go
    through tiles (the last two on both sides of that line)."""
    test_tiled_and_plain_apply_agree(prec, D, D_out, n)


@pytest.mark.parametrize("n_fit", [1, 2, 64, 511, 512, 768, 769, 1024, 2112])
@pytest.mark.parametrize("D", [5, 33, 300])
def test_statistics_around_the_few_partials_line(n_fit, D):
    """Up to twelve blocks' partials a thread adds a column's, beyond a warp: mean
    and deviation against numpy in 64 bits."""
    X = table(23 + n_fit, n_fit + 3, D)
    Y, m, s = run(X, n_fit, B.MLP_FP32, D)
    F = X[:n_fit].astype(np.float64)
    assert np.all(np.abs(m - F.mean(0)) <= 1e-12 * (np.abs(F.mean(0)) + F.std(0)))
    np.testing.assert_allclose(s, F.std(0), rtol=1e-12, atol=0)
