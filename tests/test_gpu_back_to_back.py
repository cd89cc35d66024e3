"""Calls in a row on one stream, whose kernels are launched before the last one has ended,
against the same calls each waited for: collision steps that reuse their buffers, on two
streams at once and in a graph, and training steps between changes of the weights."""

import os

import pytest
import torch

from paper_2606_15622_gb300 import api, surrogate as S

pytestmark = pytest.mark.gpu

W = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_15622_gb300", "weights")


def _inputs(n_cells, ppc, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = n_cells * ppc
    cell = torch.randint(0, n_cells, (n,), generator=g, device="cuda", dtype=torch.int32)
    v = torch.randn(3, n, generator=g, device="cuda")
    tau = 0.5 + torch.rand(n_cells, generator=g, device="cuda", dtype=torch.float64)
    return cell, v, tau


def _step(cell, v, tau, k, ws, net=None):
    return api.fp_collision_step(cell, v, tau.numel(), tau, 0.1, prec="fp32", seed=3, step=k, workspace=ws,
                                 net_lite=net)


@pytest.mark.parametrize("lite", [False, True])
@pytest.mark.parametrize("n_cells,ppc", [(37, 20), (4000, 60), (70001, 30)])
def test_steps_in_a_row(n_cells, ppc, lite):
    owner = S.Surrogate.load(os.path.join(W, "surrogate_lite.fpw"))  # (owns what net points to)
    net = owner.net() if lite else None
    ins = [_inputs(n_cells, ppc, k) for k in range(4)]
    need = api.lib().fp_collision_step_workspace_bytes(n_cells * ppc, n_cells, api.V_F32, int(lite))
    ws = torch.empty(int(need), dtype=torch.uint8, device="cuda")
    want = []
    for k, (c, v, t) in enumerate(ins):
        want.append([x.clone() for x in _step(c, v, t, k, ws, net) if x is not None])
        torch.cuda.synchronize()
    for _ in range(5):
        # the inputs of a step copied into the same buffers right before it
        c, v, t = (x.clone() for x in ins[0])
        got = []
        for k, src in enumerate(ins):
            for dst, x in zip((c, v, t), src):
                dst.copy_(x)
            got.append([x.clone() for x in _step(c, v, t, k, ws, net) if x is not None])
        for a, b in zip(want, got):
            assert all(torch.equal(x, y) for x, y in zip(a, b))


def test_steps_on_two_streams_and_in_a_graph():
    n_cells, ppc = 3000, 40
    ins = [_inputs(n_cells, ppc, k) for k in range(2)]
    need = int(api.lib().fp_collision_step_workspace_bytes(n_cells * ppc, n_cells, api.V_F32, 0))
    ws = [torch.empty(need, dtype=torch.uint8, device="cuda") for _ in range(2)]
    want = [_step(*ins[k], k, ws[k]) for k in range(2)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = [[], []]
    for _ in range(10):
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                got[k].append(_step(*ins[k], k, ws[k]))
    torch.cuda.synchronize()
    for k in range(2):
        for r in got[k]:
            assert all(torch.equal(x, y) for x, y in zip(want[k], r) if x is not None)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a = _step(*ins[0], 0, ws[0])
        b = _step(*ins[1], 1, ws[0])
    for _ in range(3):
        for x in (*a, *b):
            if x is not None:
                x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(want[0], a) if x is not None)
        assert all(torch.equal(x, y) for x, y in zip(want[1], b) if x is not None)


@pytest.mark.parametrize("batch", [64, 1000, 8192])
def test_training_steps_in_a_row(batch):
    def run(wait):
        s = S.Surrogate.load(os.path.join(W, "surrogate_full.fpw"))
        t = S.Trainer(s, batch=batch)
        g = torch.Generator(device="cuda").manual_seed(1)
        for k in range(12):
            x = torch.randn(batch, S.IN, generator=g, device="cuda").to(torch.bfloat16)
            y = torch.randn(batch, 9, generator=g, device="cuda")
            aux = torch.rand(batch, 16, generator=g, device="cuda")
            if wait:
                torch.cuda.synchronize()
            t.step(x, y, aux, 1.0 / batch)
            if k % 3 == 2:  # the weights changed by another kernel between two steps
                if wait:
                    torch.cuda.synchronize()
                s.params.mul_(0.999)
                s.shadow.mul_(0.999)
        torch.cuda.synchronize()
        return s.params.clone(), t.grads.clone(), t.m.clone(), t.v.clone()
    want = run(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(want, run(False)))
