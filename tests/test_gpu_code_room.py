"""Programs that keep an instruction for each token, in rows exactly as long: with their end marker they may have a
word more than the main passes hold.  Whichever pass takes them, their outputs have the bits of the same programs in
longer rows."""
import numpy as np
import pytest
import torch

import progtext
from paper_2603_12292_gb300 import binding as sr

pytestmark = pytest.mark.gpu

t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
UNARY = ("sin", "sqrt", "cos", "sq")


def _unfused(slots):
    """The shortest program that pushes to `slots` slots and fuses no operand into its operator."""
    if slots == 0:
        return ["x0"]
    first, second = _unfused(slots - 1), _unfused(slots - 1)
    return first + (second if slots > 1 else ["x1", "sin"]) + ["+" if slots % 2 else "-"]


def _programs(L):
    """Programs of L tokens: an unfused tree for each number of slots that fits, unary operators before and after."""
    out = []
    for slots in range(9):
        tree = _unfused(slots)
        rest = L - len(tree)
        if rest < 0:
            break
        for lead in {0, rest // 2, rest}:  # unary operators on the first leaf, the others on the result
            chain = [UNARY[i % 4] for i in range(rest)]
            out.append(progtext.parse(" ".join(tree[:1] + chain[:lead] + tree[1:] + chain[lead:])))
    assert all(len(p) == L for p in out)
    return out


def _rows(progs, Lmax):
    arr, lens = progtext.pack(progs, Lmax)
    return t(arr), t(lens)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 8, 9, 10, 16, 18, 19, 20, 38, 39, 40, 64, 71, 72, 73, 78, 79, 80, 126, 128,
                               158, 159, 160, 176, 199, 200, 201, 256, 304, 318, 319, 320, 384, 432, 510, 511])
def test_rows_as_long_as_their_programs(ctx, L):
    N = 300
    progs = _programs(L)
    X = t(np.random.default_rng(L).uniform(-3, 3, (2, 304)).astype(np.float32))
    y = t(np.random.default_rng(1).normal(size=N).astype(np.float32))
    bits = lambda x: x.clone().view({4: torch.int32, 8: torch.int64}[x.element_size()])  # noqa: E731
    want = bits(sr.sr_predict(ctx, *_rows(progs, 512), None, X, N))
    try:
        for mode in (sr.XFORM_NEVER, sr.XFORM_ALWAYS):
            sr.sr_set_transforms(ctx, mode)
            for ctas, batched in ((0, 3), (4, 4), (5, 5)):
                sr.sr_set_occupancy(ctx, ctas, batched)
                prog, lens = _rows(progs, L)
                assert torch.equal(bits(sr.sr_predict(ctx, prog, lens, None, X, N)), want), (mode, ctas)
                # the sums of one problem and of a batch over the first step (one chunk, so the same order)
                one = sr.sr_eval(ctx, prog, lens, None, X, y, 256, sr.SR_MSE)
                short = _rows([p for p in (progtext.parse("x0 x1 sin +"),)], 4)
                batch = sr.sr_eval_batched(ctx, [sr.make_problem(prog, lens, None, X, y, 256, sr.SR_MSE),
                                                 sr.make_problem(*short, None, X, y, 256, sr.SR_MSE)])
                assert torch.equal(bits(one), bits(batch[0])), (mode, batched)
    finally:
        sr.sr_set_transforms(ctx, sr.XFORM_AUTO)
        sr.sr_set_occupancy(ctx, 0, 0)
