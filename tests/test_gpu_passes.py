"""A captured call makes its later passes (programs of the extended operators, deep ones, long gradient code) only
in the replays whose own programs need them, whatever the replays before held.  Observed on the work counters at the
start of the context's workspace: a pass that was made has drawn items."""
import ctypes

import numpy as np
import pytest
import torch

import progtext
from paper_2603_12292_gb300 import binding as sr

pytestmark = pytest.mark.gpu

P, N, K, LMAX = 96, 1000, 2, 255
t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731


def _counters(ctx):
    """The first words of the workspace: its address is the fourth field of the context's struct."""
    class Struct(ctypes.Structure):
        _fields_ = [("device", ctypes.c_int), ("stream", ctypes.c_void_p), ("num_sms", ctypes.c_int),
                    ("ws", ctypes.c_void_p), ("ws_bytes", ctypes.c_size_t)]

    c = Struct.from_address(ctx.handle.value)
    assert c.device == 0 and c.num_sms == torch.cuda.get_device_properties(0).multi_processor_count
    assert c.ws_bytes >= 256

    class Words:
        __cuda_array_interface__ = {"shape": (8,), "typestr": "<i8", "data": (c.ws, False), "version": 3}

    torch.cuda.synchronize()
    return torch.as_tensor(Words(), device="cuda").cpu().tolist()


def _tree(n, op, leaf):
    """A complete binary tree of n leaves, as text."""
    return leaf if n == 1 else f"{_tree(n // 2, op, leaf)} {_tree(n // 2, op, leaf)} {op}"


BASE = "x0 x1 + sin"
KINDS = {"base": BASE, "extended": "x0 tan x1 +", "deep": _tree(64, "+", "x0 sin"),
         "long code": _tree(64, "/", "x0 c0 *")}


def _population(kind):
    texts = [BASE] * P
    texts[P // 2] = KINDS[kind]
    prog, lens = progtext.pack([progtext.parse(s) for s in texts], LMAX)
    return t(prog), t(lens)


def _replay(call, pops):
    """Captures call(ctx, programs, lengths) on a context of its own, replays it on the populations in turn; the
    counters after each."""
    prog, lens = (x.clone() for x in pops[0])
    stream = torch.cuda.Stream()
    ctx = sr.Context(0, stream)
    with torch.cuda.stream(stream):
        call(ctx, prog, lens)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            call(ctx, prog, lens)
    seen = []
    for p, n in pops:
        prog.copy_(p)
        lens.copy_(n)
        torch.cuda.synchronize()
        graph.replay()
        seen.append(_counters(ctx))
    ctx.close()
    return seen


@pytest.mark.parametrize("path", ["eval", "predict", "batched"])
def test_evaluation_passes_follow_the_replay_s_programs(path):
    c = torch.ones((P, K), device="cuda")
    X = torch.rand((2, N), device="cuda") + 1
    y = torch.rand(N, device="cuda")
    f = torch.empty(P, dtype=torch.float64, device="cuda")
    yhat = torch.empty((P, N), device="cuda")

    def call(ctx, prog, lens):
        sr.sr_set_transforms(ctx, sr.XFORM_NEVER)
        if path == "eval":
            sr.sr_eval(ctx, prog, lens, c, X, y, N, sr.SR_MSE, fitness=f)
        elif path == "predict":
            sr.sr_predict(ctx, prog, lens, c, X, N, yhat=yhat)
        else:
            sr.sr_eval_batched(ctx, [sr.make_problem(prog, lens, c, X, y, N, sr.SR_MSE, fitness=f)])

    kinds = ["base", "extended", "base", "deep", "base", "extended"]
    for kind, w in zip(kinds, _replay(call, [_population(k) for k in kinds])):
        assert w[0] > 0, kind
        assert (w[1] > 0) == (kind == "extended"), (kind, w)
        assert (w[3] > 0) == (kind == "deep"), (kind, w)
        assert w[2] == w[4] == 0, (kind, w)  # no note is left for the next call


def test_gradient_pass_follows_the_replay_s_programs():
    c = torch.full((P, K), 1.5, device="cuda")
    X = torch.rand((2, N), device="cuda") + 1
    y = torch.rand(N, device="cuda")
    mse = torch.empty(P, dtype=torch.float64, device="cuda")
    dc = torch.empty((P, K), dtype=torch.float64, device="cuda")

    def call(ctx, prog, lens):
        sr.sr_eval_grad(ctx, prog, lens, c, X, y, N, mse=mse, dconst=dc)

    kinds = ["base", "long code", "base", "long code"]
    for kind, w in zip(kinds, _replay(call, [_population(k) for k in kinds])):
        assert w[0] > 0, kind
        assert (w[1] > 0) == (kind == "long code"), (kind, w)
        assert w[2] == 0, (kind, w)
