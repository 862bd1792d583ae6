"""Self-energy buffers that the outputs overlap: the rhs is the one of separate buffers."""
import numpy as np
import pytest
import torch

from paper_1510_07799_gb300 import frg, inputs

pytestmark = pytest.mark.gpu


def case(N):
    p = frg.Params(U=1.3, T=0.64 / N, eps_d=-0.4, N_f=N)
    return (p, torch.from_numpy(inputs.random_vertex(N, p.U, seed=N)).cuda(),
            torch.from_numpy(inputs.random_sigma(N, seed=N)).cuda())


@pytest.mark.parametrize("N", [16, 26, 28, 64])
@pytest.mark.parametrize("mask", [frg.CH_ALL | frg.TAILS, frg.CH_SIGMA | frg.TAILS])
def test_tails_with_the_self_energy_rhs_in_place(N, mask):
    """The window propagators take the self-energy, not its derivative."""
    p, V, sig = case(N)
    with frg.Context([p], channel_mask=mask) as c:
        dg, ds, dg2, buf = torch.empty_like(V), torch.empty_like(sig), torch.empty_like(V), sig.clone()
        c.rhs(0, 0.25, V, sig, dg, ds)
        c.rhs(0, 0.25, V, buf, dg2, buf)
        c.stats()
        assert torch.equal(dg, dg2) and torch.equal(ds, buf)
        c.rhs_timed(0, 0.25, V, sig.clone(), dg2, ds)
        assert torch.equal(dg, dg2)


@pytest.mark.parametrize("N", [16, 26, 64])
def test_self_energy_inside_the_vertex_output(N):
    """The self-energy input may lie in the buffer that the vertex derivative fills."""
    p, V, sig = case(N)

    def check(call):
        dg, ds, dg2, ds2 = torch.empty_like(V), torch.empty_like(sig), torch.empty_like(V), torch.empty_like(sig)
        call(V, sig, dg, ds)
        torch.cuda.synchronize()
        for at in (0, N * N, N ** 3 - N):
            inner = dg2.view(-1)[at:at + N]
            inner.copy_(sig)
            call(V, inner, dg2, ds2)
            torch.cuda.synchronize()
            assert torch.equal(dg, dg2) and torch.equal(ds, ds2)
        # across the end of the vertex output and the self-energy output beside it
        both = torch.empty(N ** 3 + N, dtype=V.dtype, device="cuda")
        inner = both[N ** 3 - N // 2:N ** 3 + N // 2]
        inner.copy_(sig)
        call(V, inner, both[:N ** 3].view(N, N, N), both[N ** 3:])
        torch.cuda.synchronize()
        assert torch.equal(dg.view(-1), both[:N ** 3]) and torch.equal(ds, both[N ** 3:])

    check(lambda *a: frg.rhs_noalloc(p, 0.25, *a))
    for kw in ({}, {"precision": "3xtf32"}, {"channel_mask": frg.CH_ALL | frg.TAILS}):
        with frg.Context([p], **kw) as c:
            check(lambda *a: c.rhs(0, 0.25, *a))
