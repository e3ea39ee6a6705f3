"""Variation with half a warp per child, taken from max(8,192, 128 Lmax)
children on: children bit for bit the oracle's just below and just above the
line, for rows that a group of 16 lanes reads in one round, in several, and in
a ragged last one, with child counts that leave the last block part filled."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_12292_gb300 import binding

pytestmark = pytest.mark.gpu
CFG = dict(p_cross=0.9, p_point=0.3, p_subtree=0.3, p_const=0.5, const_delta=1.0, max_subtree=12)


@pytest.mark.parametrize("past", [-1, 0, 5])
@pytest.mark.parametrize("Lmax,K", [(1, 0), (15, 1), (16, 4), (17, 16), (33, 7), (64, 4), (68, 15), (257, 5), (512, 8)])
def test_vary_groups_bit_exact(ctx, past, Lmax, K):
    P, nv, children = 700, 4, max(8192, 128 * Lmax) + past
    prog, lens, c = oracle.random_programs(P, 1, Lmax, K, nv, -2.0, 2.0, 77, 3)
    par = np.random.default_rng(children + Lmax).integers(0, P, size=(children, 2)).astype(np.int32)
    cfg = dict(CFG, max_subtree=min(CFG["max_subtree"], Lmax))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    po, lo, co = binding.sr_vary(ctx, t(prog), t(lens), t(c) if K else None, t(par), nv, binding.var_cfg(**cfg), 99, 4)
    wp, wl, wc = oracle.vary(prog, lens, c, par, K, nv, seed=99, gen=4, **cfg)
    np.testing.assert_array_equal(lo.cpu().numpy(), wl)
    np.testing.assert_array_equal(po.cpu().numpy(), wp)
    if K:
        np.testing.assert_array_equal(co.cpu().numpy().view(np.uint32), wc.view(np.uint32))
