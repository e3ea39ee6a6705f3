"""The quotient over every binade of the divisor, from the protection's 1e-3 to the largest number, with quotients
that are subnormal, overflow or are not finite: folded constants, per-case values and variable tables agree bit for
bit, whatever the other cases of the warp divide by, and lie within 2 ulp of a / b."""
import numpy as np
import pytest
import torch

import progtext
from paper_2603_12292_gb300 import binding as sr

pytestmark = pytest.mark.gpu

t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
NEAR = np.float32(8.5e37)  # where the quotient's two forms meet


def _pairs():
    rng = np.random.default_rng(5)
    a, b = [], []
    for e in range(-11, 128):  # 2^-10 is below 1e-3: the protected ones of that binade and the next too
        lo = np.float32(2.0) ** np.float32(e)
        m = np.concatenate([[1.0, 2.0 - 2.0 ** -23], 1.0 + rng.random(10)]).astype(np.float32)
        b.append(lo * m)
    b += [np.array([1e-3, np.nextafter(np.float32(1e-3), 0, dtype=np.float32), 0.0, np.inf, np.nan], np.float32)]
    b += [np.array([NEAR, np.nextafter(NEAR, np.float32(np.inf)), np.nextafter(NEAR, np.float32(0))], np.float32)]
    b = np.concatenate(b)
    b = np.concatenate([b, -b])
    # numerators over all exponents, among them those that make the quotient subnormal or too large
    bits = rng.integers(0, 2 ** 32, 7 * len(b), dtype=np.uint32).view(np.float32)
    with np.errstate(over="ignore"):
        near = np.abs(np.resize(b, bits.size)) * np.exp2(rng.integers(-149, 128, bits.size)).astype(np.float32)
    special = np.resize(np.array([0.0, -0.0, np.inf, np.nan, 1.0, 1e-45, 3.4028235e38], np.float32), bits.size)
    a = np.concatenate([bits, near, special]).astype(np.float32)
    b = np.resize(b, a.size)
    return a, b


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("order", ["mixed", "by divisor"])
def test_every_binade_of_the_divisor(ctx, order):
    a, b = _pairs()
    p = np.random.default_rng(6).permutation(a.size) if order == "mixed" else np.argsort(np.abs(b), kind="stable")
    a, b = a[p], b[p]
    n = a.size
    X = np.zeros((2, (n + 7) // 8 * 8), np.float32)
    X[0, :n], X[1, :n] = a, b
    ulp = lambda x, y: ((x.view(np.uint32) == y.view(np.uint32)) | (np.isnan(x) & np.isnan(y)))  # noqa: E731

    def predict(texts, consts, X, N):
        prog, lens = progtext.pack([progtext.parse(s) for s in texts], 4)
        c = None if consts is None else t(consts)
        return sr.sr_predict(ctx, t(prog), t(lens), c, t(X), N).cpu().numpy()

    case, inv = predict(["x0 x1 /", "x1 inv"], None, X, n)
    # one program a pair: the pair as constants, folded by the decoder
    folded = predict(["c0 c1 /"] * n, np.stack([a, b], 1), np.ones((1, 8), np.float32), 1)[:, 0]
    assert ulp(folded, case).all(), np.nonzero(~ulp(folded, case))[0][:5]
    folded = predict(["c1 inv"] * n, np.stack([a, b], 1), np.ones((1, 8), np.float32), 1)[:, 0]
    assert ulp(folded, inv).all(), np.nonzero(~ulp(folded, inv))[0][:5]
    # one operand a constant, the other a row: a few of each kind against all cases
    at = np.linspace(0, n - 1, 97).astype(int)
    rows = predict([s for _ in at for s in ("x0 c1 /", "c0 x1 /")], np.repeat(np.stack([a[at], b[at]], 1), 2, 0), X, n)
    for k, i in enumerate(at):
        Xi = X.copy()
        Xi[1, :n] = b[i]
        assert ulp(rows[2 * k], predict(["x0 x1 /"], None, Xi, n)[0]).all(), b[i]
        Xi = X.copy()
        Xi[0, :n] = a[i]
        assert ulp(rows[2 * k + 1], predict(["x0 x1 /"], None, Xi, n)[0]).all(), a[i]
    # 1 / x_1 as a row of the variable table
    sr.sr_set_transforms(ctx, sr.XFORM_ALWAYS)
    try:
        assert ulp(predict(["x1 inv", "x1 inv"], None, X, n)[0], inv).all()
    finally:
        sr.sr_set_transforms(ctx, sr.XFORM_AUTO)

    a64, b64 = a.astype(np.float64), b.astype(np.float64)
    exact = np.where(np.abs(b) < np.float32(1e-3), 1.0, a64 / b64)
    spacing = np.maximum(np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64), 2.0 ** -149)
    fine = np.isfinite(exact) & (np.abs(exact) < 3.4028e38)
    assert (np.abs(case[fine] - exact[fine]) <= 2.0 * spacing[fine]).all()
    over = np.isfinite(exact) & (np.abs(exact) > 2.0 ** 128 * (1 + 2.0 ** -21))
    assert (case[over] == np.sign(exact[over]) * np.inf).all()
    rest = ~np.isfinite(exact)
    assert ulp(case[rest], exact[rest].astype(np.float32)).all()


def test_the_gradient_s_quotient(ctx):
    """MSE of c0 / x1 and of x0 / x1 with the numerator as a constant: what the gradient's forward pass divides is what
    the evaluation divides (one case, so that the MSE is the square of one FP32 difference)."""
    a, b = _pairs()
    keep = np.isfinite(a) & np.isfinite(b) & (np.abs(a) < 1e18) & (np.abs(a) > 1e-18)
    a, b = a[keep][::37], b[keep][::37]
    for i in range(0, a.size, 16):
        X = np.full((1, 8), b[i], np.float32)
        prog, lens = progtext.pack([progtext.parse("c0 x0 /")], 4)
        y = t(np.zeros(8, np.float32))
        c = t(np.array([[a[i]]], np.float32))
        mse, _ = sr.sr_eval_grad(ctx, t(prog), t(lens), c, t(X), y, 1)
        fit = sr.sr_eval(ctx, t(prog), t(lens), c, t(X), y, 1, sr.SR_MSE)
        assert torch.equal(mse.view(torch.int64), fit.view(torch.int64)), (a[i], b[i])
