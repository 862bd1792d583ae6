"""Evaluations whose kernels are chained (each may become resident while its
predecessor still runs): back to back on changing inputs, and recorded by a caller
(where they keep ordinary edges), they give what an evaluation by itself gives."""
import numpy as np
import pytest
import torch

from paper_1510_07799_gb300 import frg, inputs

pytestmark = pytest.mark.gpu


def params(N):
    return frg.Params(U=1.5, T=0.64 / N, eps_d=-0.5, N_f=N)


def case(N, seed):
    p = params(N)
    g = torch.from_numpy(inputs.random_vertex(N, p.U, seed=seed)).cuda()
    s = torch.from_numpy(inputs.random_sigma(N, seed=seed + 1)).cuda()
    return p, g, s


@pytest.mark.parametrize("N,precision,mask", [
    (16, "fp64", frg.CH_ALL), (32, "fp64", frg.CH_ALL), (64, "fp64", frg.CH_ALL | frg.TAILS), (82, "fp64", frg.CH_ALL),
    (34, "3xtf32", frg.CH_ALL), (66, "3xtf32", frg.CH_ALL | frg.TAILS), (50, "bf16x3", frg.CH_ALL)])
def test_back_to_back_and_captured(N, precision, mask):
    ins = [case(N, 10 + 3 * i) for i in range(4)]
    outs = [(torch.empty_like(g), torch.empty_like(s)) for _, g, s in ins]
    st = torch.cuda.Stream()
    with frg.Context([ins[0][0]], precision=precision, channel_mask=mask, stream=st.cuda_stream) as c:
        alone = []
        for i, (_, g, s) in enumerate(ins):
            c.rhs(0, 0.1 + 0.2 * i, g, s, *outs[i])
            st.synchronize()
            alone.append([x.cpu().numpy().copy() for x in outs[i]])
        for _ in range(20):
            for x in outs:
                x[0].zero_()
            torch.cuda.synchronize()
            for i, (_, g, s) in enumerate(ins):
                c.rhs(0, 0.1 + 0.2 * i, g, s, *outs[i])
            st.synchronize()
            for a, x in zip(alone, outs):
                assert np.array_equal(a[0], x[0].cpu().numpy()) and np.array_equal(a[1], x[1].cpu().numpy())
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            for i, (_, g, s) in enumerate(ins):
                c.rhs(0, 0.1 + 0.2 * i, g, s, *outs[i])
        for _ in range(3):
            for x in outs:
                x[0].zero_()
            graph.replay()
        torch.cuda.synchronize()
        for a, x in zip(alone, outs):
            assert np.array_equal(a[0], x[0].cpu().numpy()) and np.array_equal(a[1], x[1].cpu().numpy())
