"""The merge of a program's case chunks, a group of lanes per program by the
number of chunks: both fitness kinds, single and batched, around the group
sizes, against FP64 sums of the program outputs."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding, inputs
from progtext import pack, parse

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunks", [1, 2, 4, 5, 8, 9, 17, 33, 64, 65, 128, 129, 300])
def test_fitness_for_any_number_of_chunks(ctx, chunks):
    rng = np.random.default_rng(chunks)
    N = 256 * chunks - (37 if chunks > 1 else 200)  # a ragged last chunk
    X = rng.uniform(1, 3, (2, (N + 3) // 4 * 4)).astype(np.float32)
    texts = ["x0 x1 +", "x0 x1 *", "x0 sq x1 -", "x1 c0 * x0 -", "x0 sin x1 +", "c0", "x0 exp", "+"]
    texts = texts * 9  # more programs than one block merges
    progs, lens = pack([parse(t) for t in texts], 6)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    c = t(np.full((len(texts), 1), 0.75, np.float32))
    y = (X[0, :N] * X[1, :N] + rng.normal(0, 0.5, N)).astype(np.float32)
    args = (t(progs), t(lens), c, t(X), t(y), N)
    out = binding.sr_predict(ctx, args[0], args[1], c, args[3], N).cpu().numpy().astype(np.float64)
    binding.sr_set_tile(ctx, 256)
    try:
        got = binding.sr_eval(ctx, *args, binding.SR_MSE_CORR).cpu().numpy()
    finally:
        binding.sr_set_tile(ctx, 0)
    probs = [binding.make_problem(*args, k, cases_per_tile=256) for k in (binding.SR_MSE, binding.SR_CORR)]
    batched = torch.stack(binding.sr_eval_batched(ctx, probs)).cpu().numpy()
    assert np.array_equal(got, batched)  # the same chunks, the same sums
    y64 = y.astype(np.float64)
    for p, text in enumerate(texts):
        if text == "+":
            assert np.isinf(got[:, p]).all()
            continue
        # FP32 errors, squares and 8-case sums round a handful of times: 2^-20 of sums of positive
        # terms; r^2 takes four such sums
        mse = np.mean((out[p] - y64) ** 2)
        assert abs(got[0, p] - mse) <= 2.0 ** -20 * mse, (text, p)
        want = 1.0 if text == "c0" else 1.0 - np.corrcoef(out[p], y64)[0, 1] ** 2
        assert abs(got[1, p] - want) <= 2.0 ** -17, (text, p)


@pytest.mark.parametrize("tile", [256, 2560, 2816, 6144])
def test_batched_items_short_and_long_equal_single_calls(ctx, tile):
    """Both copies of the batched kernel (short and long items) against sr_eval with the same chunks."""
    rng = np.random.default_rng(tile)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    probs, single = [], []
    binding.sr_set_tile(ctx, tile)
    try:
        for i, N in enumerate((6144, 6001, 12_288)):
            pr = inputs.make_problem("items", 70 + i, P=90, Lmin=1, Lmax=40, nvars=3, K=2, N=N, xlo=-2.0, xhi=2.0,
                                     target_len=(3, 7), unary_ops=12 if i == 1 else 6)
            y = t(rng.normal(0, 1, N).astype(np.float32))
            args = (t(pr.programs), t(pr.lengths), t(pr.consts), t(pr.X), y, N, binding.SR_MSE_CORR)
            single.append(binding.sr_eval(ctx, *args))
            probs.append(binding.make_problem(*args, cases_per_tile=tile))
        got = binding.sr_eval_batched(ctx, probs)
    finally:
        binding.sr_set_tile(ctx, 0)
    for a, b in zip(got, single):
        assert torch.equal(a, b)
