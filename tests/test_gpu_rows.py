"""How the interpreter reads rows of X: a 256-bit load per lane where the rows
allow it (their own layout, a copy, or the variable table), 128-bit halves
where there is no room for a copy.  Every layout gives the same bits.  Also
the operators whose range test is made once for eight values: lanes that mix
arguments inside and outside the common range."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding, inputs
from progtext import pack, parse

pytestmark = pytest.mark.gpu


def _problem(N, unary_ops=inputs.UNARY_ALL, P=96, Lmax=48, nvars=5, K=3):
    pr = inputs.make_problem("rows", 900 + N, P=P, Lmin=1, Lmax=Lmax, nvars=nvars, K=K, N=N, xlo=-3.0, xhi=3.0,
                             target_len=(3, 7), unary_ops=unary_ops)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    y = t(np.cos(pr.X[0, :N]).astype(np.float32))
    return pr, t(pr.programs), t(pr.lengths), t(pr.consts), t(pr.X), y


def _layout(X, N, ldx, offset):
    """X's first N columns with row stride ldx, `offset` floats into a buffer."""
    buf = torch.full((X.shape[0] * ldx + offset,), 7.0, device="cuda")
    out = buf[offset:].view(X.shape[0], ldx)
    out[:, :N] = X[:, :N]
    return out


@pytest.mark.parametrize("N", [1, 4, 7, 8, 9, 255, 257, 1020, 4100])
def test_every_row_layout_gives_the_same_bits(ctx, N):
    pr, prog, lens, cons, X, y = _problem(N)
    up8, up4 = (N + 7) // 8 * 8, (N + 3) // 4 * 4
    odd = up4 if up4 % 8 else up4 + 4  # a stride that is no multiple of 8
    binding.sr_set_transforms(ctx, 0)
    try:
        got = []
        for ldx, off in ((up8, 0), (up8, 4), (odd, 0), (odd, 4)):
            Xl = _layout(X, N, ldx, off)
            got.append((binding.sr_predict(ctx, prog, lens, cons, Xl, N),
                        binding.sr_eval(ctx, prog, lens, cons, Xl, y, N, binding.SR_MSE_CORR),
                        binding.sr_eval_batched(ctx, [binding.make_problem(prog, lens, cons, Xl, y, N, k)
                                                      for k in (0, 1)])[1].clone()))
        torch.cuda.synchronize()
    finally:
        binding.sr_set_transforms(ctx, 1)
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


def test_a_captured_call_without_room_for_a_copy_reads_halves():
    N = 60_004
    pr, prog, lens, cons, X, y = _problem(N, P=8, nvars=16, Lmax=200)
    ctx = binding.Context(0)
    try:
        binding.sr_set_transforms(ctx, 0)
        wide = _layout(X, N, (N + 7) // 8 * 8, 0)
        want = binding.sr_eval(ctx, prog, lens, cons, wide, y, N, binding.SR_MSE_CORR).clone()
        torch.cuda.synchronize()
        odd = _layout(X, N, N, 0)  # 60,004 = 4 mod 8: would be copied, 3.8 MB more than the workspace holds
        probs = [binding.make_problem(prog, lens, cons, odd, y, N, binding.SR_MSE)]
        out = torch.zeros_like(want)
        stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        ctx.set_stream(stream)
        with torch.cuda.graph(g, stream=stream):
            binding.sr_eval(ctx, prog, lens, cons, odd, y, N, binding.SR_MSE_CORR, fitness=out)
            mse = binding.sr_eval_batched(ctx, probs)[0]
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want.cpu().numpy(), equal_nan=True)
        # the batch cuts its own case chunks: FP32 compensated sums of the same errors, to a few
        # roundings of a chunk's largest term (2^-22 of the sum at most)
        a, b = mse.cpu().numpy(), want[0].cpu().numpy()
        assert np.array_equal(np.isfinite(a), np.isfinite(b))
        ok = np.isfinite(b)
        assert (np.abs(a[ok] - b[ok]) <= 2.0 ** -22 * np.abs(b[ok])).all()
    finally:
        ctx.close()


def test_noalloc_reads_rows_of_any_layout(ctx):
    N = 1021
    pr, prog, lens, cons, X, y = _problem(N)
    binding.sr_set_transforms(ctx, 0)
    try:
        want = binding.sr_eval(ctx, prog, lens, cons, _layout(X, N, 1024, 0), y, N, binding.SR_MSE_CORR)
    finally:
        binding.sr_set_transforms(ctx, 1)
    for ldx, off in ((1024, 0), (1028, 0), (1024, 4)):
        out = torch.zeros_like(want)
        assert binding.sr_eval_noalloc(prog, lens, cons, _layout(X, N, ldx, off), y, N, 2, out) == binding.SR_OK
        assert torch.equal(out, want)


def test_mixed_ranges_within_a_lane(ctx):
    """sin, cos and the quotient where some of a lane's eight arguments leave
    the common range: FP64 references, 2 ulp (2^-22 relative, 2^-148 absolute),
    NaN and infinities where the real function has them."""
    rng = np.random.default_rng(5)
    N = 2048
    X = rng.uniform(-6, 6, (2, N)).astype(np.float32)
    far = rng.random((2, N)) < 0.15
    X[far] = (rng.choice([-1, 1], far.sum()) * 10.0 ** rng.uniform(4.5, 38.4, far.sum())).astype(np.float32)
    X[0, :5] = [np.inf, -np.inf, np.nan, 4.0e4, -4.0001e4]
    X[1, 5:11] = [np.inf, np.nan, 8.5e37, 8.51e37, 1e-3, 0.99e-3]
    # x * 1 keeps the operand out of the variable table
    progs, lens = pack([parse(t) for t in ("x0 c0 * sin", "x0 c0 * cos", "x0 c0 * x1 /", "x1 c0 * x0 x1 - c1 * /")], 12)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = binding.sr_predict(ctx, t(progs), t(lens), t(np.tile(np.float32([1, 0]), (4, 1))), t(X), N).cpu().numpy()
    a, b = X.astype(np.float64)
    with np.errstate(all="ignore"):
        zero = (X[0] - X[1]) * np.float32(0)  # 0, or NaN where x0 - x1 is not finite
        quot = lambda p, q: np.where(np.abs(q) < np.float64(np.float32(1e-3)), 1.0, p / q)
        want = [np.sin(a), np.cos(a), quot(a, b), quot(b, zero.astype(np.float64))]
    for k, w in enumerate(want):
        g = got[k].astype(np.float64)
        big = np.abs(w) >= 2.0 ** 128 * (1 - 2.0 ** -25)
        assert np.array_equal(np.isnan(g), np.isnan(w)), k
        assert (np.isinf(g) | (np.abs(g) > 3.4e38))[big & ~np.isnan(w)].all(), k
        fine = ~np.isnan(w) & ~big
        assert (np.abs(g - w)[fine] <= 2.0 ** -22 * np.abs(w[fine]) + 2.0 ** -148).all(), k
