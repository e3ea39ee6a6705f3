"""The gradient of programs whose operators see NaN: the value and the partial are NaN, alone in a warp, in all of
it, or beside an argument beyond the moderate range of sin and cos.  The MSE is then the worst, as the evaluation
has it, and the derivative NaN, as FP64 autograd has it."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding

pytestmark = pytest.mark.gpu

FUNCTIONS = {4: torch.sin, 5: torch.cos, 6: torch.exp, 7: lambda x: x.abs().log(),
             8: lambda x: x.abs().sqrt(), 9: torch.square, 10: torch.reciprocal, 11: torch.tan, 12: torch.asin,
             13: torch.acos, 14: torch.atan, 15: torch.tanh}


@pytest.mark.parametrize("where", ["one", "all", "beside far"])
def test_a_nan_argument_gives_nan(ctx, where):
    N = 300
    x = torch.full((1, N), 0.25, device="cuda")
    if where == "all":
        x[:] = torch.inf
    else:
        x[0, 5] = torch.inf
    far = torch.zeros_like(x)
    if where == "beside far":
        far[0, 9] = 1.0e5
    X = torch.cat([x, far]).contiguous()
    y = torch.zeros(N, device="cuda")
    # f(((x0 - x0) + x1) + c0): x0 - x0 is NaN where x0 is infinite
    toks = [[16, 16, 1, 17, 0, 32, 0, op] for op in FUNCTIONS]
    prog = torch.tensor(toks, dtype=torch.uint8, device="cuda")
    lens = torch.full((len(toks),), len(toks[0]), dtype=torch.int32, device="cuda")
    c = torch.full((len(toks), 1), 0.5, device="cuda")
    mse, dconst = binding.sr_eval_grad(ctx, prog, lens, c, X, y, N)
    plain = binding.sr_eval(ctx, prog, lens, c, X, y, N, binding.SR_MSE)
    torch.cuda.synchronize()
    for i, f in enumerate(FUNCTIONS.values()):
        k = torch.tensor(0.5, dtype=torch.float64, requires_grad=True)
        xd = X.double().cpu()
        loss = (f(xd[0] - xd[0] + xd[1] + k) ** 2).mean()
        (want,) = torch.autograd.grad(loss, k)
        assert torch.isnan(loss) and torch.isnan(want), i
    assert np.all(np.isposinf(plain.cpu().numpy()))
    assert np.all(np.isposinf(mse.cpu().numpy()))
    assert np.all(np.isnan(dconst.cpu().numpy()))
