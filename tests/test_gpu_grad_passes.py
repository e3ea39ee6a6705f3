"""The gradient's second pass, for programs whose code outgrows a warp's share of shared memory: made only where a
program can be so long, and with the bits of the first pass whichever takes a program.  And its slices, where the
workspace has no room for the whole call and cannot grow."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding as sr
from paper_2603_12292_gb300 import inputs

pytestmark = pytest.mark.gpu

t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731


def _problem(P, Lmax, K, N=700, seed=3):
    pr = inputs.make_problem("passes", seed, P=P, Lmin=1, Lmax=Lmax, nvars=3, K=K, N=N, xlo=1.0, xhi=5.0,
                             target_len=(5, 9))
    y = np.sin(pr.X[0, :N]) + pr.X[1, :N]
    return t(pr.programs), t(pr.lengths), t(pr.consts), t(pr.X), t(y.astype(np.float32)), N


# the code of 70 tokens (at most 319 words) fits beside 4 CTAs per SM at 8 constants, that of 72 does not
@pytest.mark.parametrize("Lmax,K,passes", [(1, 1, 1), (24, 8, 1), (64, 2, 1), (64, 8, 1), (70, 8, 1), (72, 8, 2), (128, 8, 2),
                                           (255, 4, 2), (512, 2, 2)])
@pytest.mark.parametrize("batched", [False, True])
def test_launches(ctx, Lmax, K, passes, batched):
    prog, lens, c, X, y, N = _problem(40, Lmax, K)
    before = sr.sr_kernel_launches(ctx)
    if batched:
        sr.sr_eval_grad_batched(ctx, [sr.make_grad_problem(prog, lens, c, X, y, N)])
    else:
        sr.sr_eval_grad(ctx, prog, lens, c, X, y, N)
    sr.sr_sync(ctx)
    assert sr.sr_kernel_launches(ctx) - before == 2 + passes  # decoding, the passes, the merge


def test_the_launch_s_layout_does_not_change_results(ctx):
    """A batch is laid out for its longest rows and most constants, so that a program may take another pass than in
    a call of its own: the results keep their bits."""
    probs = [_problem(60, L, K, seed=5 + L) for L, K in ((16, 8), (64, 2), (128, 8), (200, 16), (512, 4))]
    alone = [sr.sr_eval_grad(ctx, *p) for p in probs]
    batch = sr.sr_eval_grad_batched(ctx, [sr.make_grad_problem(*p) for p in probs])
    sr.sr_sync(ctx)
    for a, b in zip(alone, batch):
        for u, v in zip(a, b):
            assert torch.equal(u.view(torch.int64), v.view(torch.int64))


def _captured(warm, problems, batched):
    """The gradients of problems from a call captured on a context whose workspace one call on `warm` has sized, and
    the kernels it launched."""
    out = [(torch.empty(p[0].shape[0], dtype=torch.float64, device="cuda"),
            torch.empty(p[2].shape, dtype=torch.float64, device="cuda")) for p in problems]
    stream = torch.cuda.Stream()
    ctx = sr.Context(0, stream)
    with torch.cuda.stream(stream):
        sr.sr_eval_grad(ctx, *warm)
        torch.cuda.synchronize()
        before = sr.sr_kernel_launches(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            if batched:
                sr.sr_eval_grad_batched(ctx, [sr.make_grad_problem(*p, mse=m, dconst=d)
                                              for p, (m, d) in zip(problems, out)])
            else:
                for p, (m, d) in zip(problems, out):
                    sr.sr_eval_grad(ctx, *p, mse=m, dconst=d)
        launches = sr.sr_kernel_launches(ctx) - before
        for _ in range(2):
            graph.replay()
    torch.cuda.synchronize()
    ctx.close()
    return out, launches


def _many(ctx, P, Lmax, K, nvars, N):
    """P random programs, drawn on the GPU."""
    prog, lens, c = sr.sr_random_programs(ctx, P, 1, Lmax, K, nvars, -5.0, 5.0, 99, 7)
    X = torch.rand((nvars, N), device="cuda") * 4 + 1
    return prog, lens, c, X, torch.sin(X[0]) + X[nvars - 1], N


# a workspace sized by 256 programs of 64 tokens holds the tapes but not the code of 40,000; one sized by 4 tokens
# holds neither the tapes nor the code of 300 programs of 64
@pytest.mark.parametrize("P,Lmax,warmP,warmL", [(40_000, 64, 256, 64), (300, 64, 256, 4), (1, 64, 1, 1)])
@pytest.mark.parametrize("batched", [False, True])
def test_a_captured_call_in_a_small_workspace(ctx, P, Lmax, warmP, warmL, batched):
    problems = [_many(ctx, P, Lmax, 4, 3, 600)]
    if batched:
        problems.append(_many(ctx, 77, 16, 2, 3, 300))
    want = [sr.sr_eval_grad(ctx, *p) for p in problems]
    got, launches = _captured(_many(ctx, warmP, warmL, 4, 3, 600), problems, batched)
    sr.sr_sync(ctx)
    if P > 10_000:
        assert launches > 3 * len(problems)
    for a, b in zip(want, got):
        for u, v in zip(a, b):
            assert torch.equal(u.view(torch.int64), v.view(torch.int64))
