"""The decoders, a warp per program in blocks of 32 tokens: programs whose
lengths lie around the block edges, chains and balanced trees, invalid bytes on
either side of an edge; and the adjoint's second pass, for programs whose code
outgrows the first one's share of shared memory."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_12292_gb300 import binding, inputs
from progtext import pack, parse

pytestmark = pytest.mark.gpu

EDGES = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 511, 512]


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _evaluate(tok, c, X):
    """+ - * and squares in FP32, each rounded once: what any order of evaluation gives."""
    st = []
    for v in tok:
        if v >= 32:
            st.append(np.full(X.shape[1], c[v - 32]))
        elif v >= 16:
            st.append(X[v - 16])
        elif v == 9:
            st.append(st[-1] * st.pop())
        else:
            b, a = st.pop(), st.pop()
            st.append(a + b if v == 0 else a - b if v == 1 else a * b)
    return st[0]


@pytest.mark.parametrize("L", EDGES)
def test_lengths_around_the_blocks_of_32(ctx, L):
    rng = np.random.default_rng(L)
    N, nvars, K, Lmax = 70, 4, 3, max(L, 4)
    prog, lens = inputs.random_programs(rng, 40, L, L, nvars, K, width=Lmax, unary_tokens=[9], binary_tokens=[0, 1, 2])
    rows = [prog[p] for p in range(40)]
    chain = np.zeros(Lmax, np.uint8)  # a variable, then squares: the longest chain
    chain[:L] = 9
    chain[0] = 16
    right = np.zeros(Lmax, np.uint8)  # x0 x1 ... - - -: every left operand far back
    m = (L + 1) // 2
    right[:m], right[m:2 * m - 1] = 16 + np.arange(m) % nvars, 1
    left = np.zeros(Lmax, np.uint8)   # x0 x1 - x2 - ...
    left[:2 * m - 1] = 1
    left[:1], left[1:2 * m - 1:2] = 16, 16 + np.arange(1, m) % nvars
    rows += [chain, right, left]
    lens = np.concatenate([lens, [L, 2 * m - 1, 2 * m - 1]]).astype(np.int32)
    prog = np.stack(rows)
    X = rng.uniform(-1.2, 1.2, (nvars, 72)).astype(np.float32)
    c = rng.uniform(-1.2, 1.2, (len(prog), K)).astype(np.float32)
    for mode in (0, 2):
        binding.sr_set_transforms(ctx, mode)
        try:
            got = binding.sr_predict(ctx, _t(prog), _t(lens), _t(c), _t(X), N).cpu().numpy()
        finally:
            binding.sr_set_transforms(ctx, 1)
        with np.errstate(all="ignore"):
            want = np.stack([_evaluate(prog[p, :lens[p]], c[p], X[:, :N]) for p in range(len(prog))])
        assert np.array_equal(got, want, equal_nan=True)


def test_flags_around_the_blocks_of_32(ctx):
    rng = np.random.default_rng(3)
    P, Lmax, nvars, K = 400, 130, 3, 2
    prog, lens = inputs.random_programs(rng, P, 1, Lmax, nvars, K)
    for p in range(P):  # damage at an edge of a block, or anywhere
        t = int(rng.choice([0, 31, 32, 33, 63, 64, 65, 95, 96, 127, 128, int(rng.integers(Lmax))]))
        prog[p, t % lens[p]] = rng.choice([0, 4, 9, 16, 16 + nvars, 32, 32 + K, 50, 200])
    lens[:3] = [0, Lmax + 1, -7]
    N = 9
    X, y = np.ones((nvars, 12), np.float32), np.ones(N, np.float32)
    want = oracle.validate_all(prog, lens, nvars, K)[0]
    c = np.ones((P, K), np.float32)
    for call in ("eval", "grad"):
        flags = torch.full((P,), -1, dtype=torch.int32, device="cuda")
        if call == "eval":
            binding.sr_eval(ctx, _t(prog), _t(lens), _t(c), _t(X), _t(y), N, binding.SR_MSE, prog_flags=flags)
        else:
            binding.sr_eval_grad(ctx, _t(prog), _t(lens), _t(c), _t(X), _t(y), N, prog_flags=flags)
        assert np.array_equal(flags.cpu().numpy(), want), call


def _quotients(n):
    """A balanced tree of n quotients' operands c x +: 2.5 code words a token, more than the main pass keeps."""
    if n == 1:
        return "c0 x0 +"
    return f"{_quotients(n // 2)} {_quotients(n - n // 2)} /"


def test_the_second_pass_gives_the_first_ones_bits(ctx):
    texts = [_quotients(n).replace("c0", f"c{n % 3}") for n in (2, 5, 12, 16)]
    L = max(len(t.split()) for t in texts)
    rng = np.random.default_rng(4)
    N = 300
    X, y = rng.uniform(1, 3, (1, 300)).astype(np.float32), rng.uniform(1, 3, N).astype(np.float32)
    c = rng.uniform(1, 3, (len(texts), 3)).astype(np.float32)
    got = []
    for Lmax in (L, 3 * L):  # at 3 L every program fits the main pass
        progs, lens = pack([parse(t) for t in texts], Lmax)
        got.append(binding.sr_eval_grad(ctx, _t(progs), _t(lens), _t(c), _t(X), _t(y), N))
        got.append(binding.sr_eval_grad_batched(ctx, [binding.make_grad_problem(_t(progs), _t(lens), _t(c), _t(X), _t(y),
                                                                                N)])[0])
    torch.cuda.synchronize()
    for mse, dc in got[1:]:
        assert torch.equal(mse, got[0][0]) and torch.equal(dc, got[0][1])
    g = oracle.grad(*pack([parse(t) for t in texts], L), c, X, y, N)
    ref, scale = np.asarray(g[1]), np.asarray(g[3])
    assert (np.abs(got[0][1].cpu().numpy() - ref) <= 2e-4 * scale).all()
