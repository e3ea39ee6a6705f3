"""Rows of X that cannot be read by 256-bit loads, where there is no room to copy them: the call makes the passes
that it makes with room (base operators, extended ones, deep programs), and gives the same bits."""
import numpy as np
import pytest
import torch

from paper_2603_12292_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lmax,ops", [(64, inputs.N_UNARY), (64, inputs.UNARY_ALL), (256, inputs.UNARY_ALL)])
def test_the_passes_are_those_of_a_call_with_room(Lmax, ops):
    N, P, nvars = 60_004, 8, 16  # 60,004 = 4 mod 8: X would be copied
    pr = inputs.make_problem("halves", 31 + Lmax, P=P, Lmin=Lmax // 2, Lmax=Lmax, nvars=nvars, K=3, N=N, xlo=-3.0,
                             xhi=3.0, target_len=(3, 7), unary_ops=ops)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    prog, lens, cons, y = t(pr.programs), t(pr.lengths), t(pr.consts), t(np.cos(pr.X[0, :N]).astype(np.float32))
    X = t(pr.X[:, :N])

    def calls(ctx, out):
        binding.sr_set_transforms(ctx, 0)
        probs = [binding.make_problem(prog, lens, cons, X, y, N, k, fitness=out[i + 1]) for i, k in enumerate((0, 1))]
        n = [binding.sr_kernel_launches(ctx)]
        binding.sr_eval(ctx, prog, lens, cons, X, y, N, binding.SR_CORR, fitness=out[0])
        n.append(binding.sr_kernel_launches(ctx))
        binding.sr_eval_batched(ctx, probs)
        n.append(binding.sr_kernel_launches(ctx))
        return np.diff(n).tolist()

    want, got = (torch.zeros((3, P), dtype=torch.float64, device="cuda") for _ in range(2))
    roomy, tight = binding.Context(0), binding.Context(0)
    try:
        launches = calls(roomy, want)
        # a workspace for the calls without the copies (3.8 MB each): that of wide rows
        wide = torch.zeros((nvars, 60_008), device="cuda")
        wide[:, :N] = X
        binding.sr_set_transforms(tight, 0)
        binding.sr_eval(tight, prog, lens, cons, wide, y, N, binding.SR_CORR, fitness=got[0])
        binding.sr_eval_batched(tight, [binding.make_problem(prog, lens, cons, wide, y, N, k, fitness=got[i + 1])
                                        for i, k in enumerate((0, 1))])
        got.zero_()
        torch.cuda.synchronize()
        stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        tight.set_stream(stream)
        with torch.cuda.graph(g, stream=stream):
            captured = calls(tight, got)
        g.replay()
        torch.cuda.synchronize()
        assert captured == launches
        assert torch.equal(got, want)
    finally:
        roomy.close()
        tight.close()
