"""Calls queued one after the other without a wait between them, whose kernels overlap, give the bits of calls that
are waited for: buffers and workspace that change from call to call are read as the call before left them."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding as sr
from paper_2603_12292_gb300 import inputs

pytestmark = pytest.mark.gpu

t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731


def _problem(seed, P=48, N=1004, nvars=4, K=3, Lmax=24):
    pr = inputs.make_problem("chain", seed, P=P, Lmin=1, Lmax=Lmax, nvars=nvars, K=K, N=N, xlo=-4.0, xhi=4.0,
                             target_len=(5, 9))
    y = np.cos(pr.X[0, :N]) * (1 + seed % 5) + pr.X[1 % nvars, :N]
    return t(pr.programs), t(pr.lengths), t(pr.consts), t(pr.X), t(y.astype(np.float32))


def _bits(x):
    return x.view({1: torch.uint8, 4: torch.int32, 8: torch.int64}[x.element_size()])


def _same(a, b):
    assert len(a) == len(b)
    for i, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(_bits(x), _bits(y)), i


def _queued_and_waited(calls):
    """The outputs of calls(wait) without and with a wait after each call."""
    torch.cuda.synchronize()
    queued = calls(lambda: None)
    torch.cuda.synchronize()
    waited = calls(torch.cuda.synchronize)
    torch.cuda.synchronize()
    return queued, waited


@pytest.mark.parametrize("N", [1004, 1000])  # rows that are copied into the workspace, rows read in place
@pytest.mark.parametrize("mode", [sr.XFORM_NEVER, sr.XFORM_ALWAYS])
def test_evaluations_of_changing_data(N, mode):
    ctx = sr.Context(0)
    sr.sr_set_transforms(ctx, mode)
    probs = [_problem(s, N=N) for s in (1, 2, 3)]
    P = probs[0][0].shape[0]
    X, y = torch.empty_like(probs[0][3]), torch.empty_like(probs[0][4])

    def calls(wait):
        out = []
        for i in range(48):
            prog, lens, c, Xi, yi = probs[i % 3]
            if i % 2:  # the same buffers with other data, written by ordinary launches
                X.copy_(Xi)
                y.copy_(yi)
                Xi, yi = X, y
            f = torch.empty((2, P), dtype=torch.float64, device="cuda")
            s = torch.empty(P, dtype=torch.float64, device="cuda")
            sr.sr_eval(ctx, prog, lens, c, Xi, yi, N, sr.SR_MSE_CORR, fitness=f)
            wait()
            sr.sr_eval_score(ctx, prog, lens, c, Xi, yi, N, sr.SR_SCORE_R4, 100, score=s)
            wait()
            out += [f, s]
        return out

    _same(*_queued_and_waited(calls))
    ctx.close()


def test_outputs_as_the_next_call_s_variables():
    ctx = sr.Context(0)
    N = 1008
    prog, lens, c, X, y = _problem(7, P=60, N=N)
    yhat = torch.empty((4, N), dtype=torch.float32, device="cuda")

    def calls(wait):
        out = []
        for i in range(40):
            f = torch.empty(60, dtype=torch.float64, device="cuda")
            k = 4 * (i % 15)
            sr.sr_predict(ctx, prog[k:k + 4], lens[k:k + 4], c[k:k + 4], X, N, yhat=yhat)
            wait()
            sr.sr_eval(ctx, prog, lens, c, yhat, yhat[i % 4], N, sr.SR_CORR, fitness=f)
            wait()
            out.append(f)
        return out

    _same(*_queued_and_waited(calls))
    ctx.close()


@pytest.mark.parametrize("P,Lmax", [(96, 24), (8192, 32), (200, 33)])
def test_selection_and_variation_on_two_buffers(P, Lmax):
    ctx = sr.Context(0)
    prog, lens, c, _, _ = _problem(11, P=P, Lmax=Lmax)
    cfg = sr.var_cfg(max_subtree=8)
    fit = [torch.rand(P, dtype=torch.float64, device="cuda") for _ in range(2)]

    def calls(wait):
        a = (prog.clone(), lens.clone(), c.clone())
        b = tuple(torch.empty_like(x) for x in a)
        par = torch.empty((P, 2), dtype=torch.int32, device="cuda")
        for g in range(60):
            sr.sr_select_tournament(ctx, fit[g & 1], 4, 5, g, parents=par)
            wait()
            sr.sr_vary(ctx, *a, par, 4, cfg, 5, g, out=b)
            wait()
            a, b = b, a
        return list(a) + [par]

    _same(*_queued_and_waited(calls))
    ctx.close()


def test_generations_and_adam_steps():
    ctx = sr.Context(0)
    N, P = 1004, 64
    prog, lens, c, X, y = _problem(13, P=P, N=N)
    cfg, adam = sr.var_cfg(max_subtree=6), sr.adam_cfg()

    def calls(wait):
        a = (prog.clone(), lens.clone(), c.clone())
        b = tuple(torch.empty_like(x) for x in a)
        par = torch.empty((P, 2), dtype=torch.int32, device="cuda")
        f = torch.empty(P, dtype=torch.float64, device="cuda")
        mse, dc = torch.empty_like(f), torch.empty((P, c.shape[1]), dtype=torch.float64, device="cuda")
        m, v = torch.zeros_like(dc), torch.zeros_like(dc)
        out = []
        for g in range(12):
            for s in range(2):
                sr.sr_eval_grad(ctx, *a, X, y, N, mse=mse, dconst=dc)
                wait()
                sr.sr_adam_step(ctx, a[2], dc, m, v, 2 * g + s + 1, adam)
                wait()
            sr.sr_eval(ctx, *a, X, y, N, sr.SR_CORR, fitness=f)
            wait()
            sr.sr_select_tournament(ctx, f, 4, 9, g, parents=par)
            wait()
            sr.sr_vary(ctx, *a, par, 4, cfg, 9, g, out=b)
            wait()
            out += [f.clone(), mse.clone(), dc.clone()]
            a, b = b, a
        return out + list(a)

    _same(*_queued_and_waited(calls))
    ctx.close()
