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
