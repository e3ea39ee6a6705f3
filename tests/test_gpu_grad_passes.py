"""The gradient's second pass, for programs whose code outgrows a warp's share of shared memory: made only where a
program can be so long, and with the bits of the first pass whichever takes a program."""
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
