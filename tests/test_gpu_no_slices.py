"""FP64 contexts whose sliced operands find no room: the channel products on the CUDA
cores, against the oracle and against the sliced products."""
import contextlib

import numpy as np
import pytest

import oracle
from paper_1510_07799_gb300 import frg, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12  # the FP64 path's bar for one rhs
FLOW_TOL = 1e-10  # and for a flow


@contextlib.contextmanager
def no_slices():
    frg.load().frg_selftest_slices(0)
    try:
        yield
    finally:
        frg.load().frg_selftest_slices(1)


def params(N, U=1.3):
    return frg.Params(U=U, T=0.64 / N, eps_d=-0.4, N_f=N)


def nrel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


@pytest.mark.parametrize("mask", [0xF, 0x1, 0x2, 0xC, 0xF | frg.TAILS])
@pytest.mark.parametrize("N", [28, 32, 66])
def test_rhs_matches_oracle(N, mask):
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=N + mask, crossing=False)
    sig = inputs.random_sigma(N, seed=N)
    g, s = torch.from_numpy(V).cuda(), torch.from_numpy(sig).cuda()
    dg, ds = torch.empty_like(g), torch.empty_like(s)
    with no_slices(), frg.Context([p], channel_mask=mask) as c:
        n0 = frg.kernel_launches()
        c.rhs(0, 0.25, g, s, dg, ds)
        launches = frg.kernel_launches() - n0
        c.stats()
    with frg.Context([p], channel_mask=mask) as c:  # (three kernels for all channels)
        n0 = frg.kernel_launches()
        c.rhs(0, 0.25, g, s, dg.clone(), ds.clone())
        assert frg.kernel_launches() - n0 - launches == 3 - bin(mask & 7).count("1")
        c.stats()
    rg, rs = oracle.rhs(oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N), 0.25, V, sig, mask=mask)
    assert nrel(dg.cpu().numpy(), rg) < TOL
    if mask & 8:
        assert nrel(ds.cpu().numpy(), rs) < TOL


def flow(pts, mask):
    with frg.Context(pts, channel_mask=mask) as c:
        st = c.flow()
        return [[x.cpu().numpy() for x in c.get_state(i)[:2]] for i in range(len(pts))], [x.accepted for x in st]


@pytest.mark.parametrize("extra", [0, frg.NO_REVERSAL])
def test_flows_match_the_sliced_ones(extra):
    """Mixed with grids of the one-launch rhs."""
    pts = [params(n, U=1.0 + 0.1 * i) for i, n in enumerate((16, 30, 8, 40))]
    with no_slices():
        a, na = flow(pts, frg.CH_ALL | extra)
    b, nb = flow(pts, frg.CH_ALL | extra)
    assert na == nb
    for x, y in zip(a, b):
        assert nrel(x[0], y[0]) < FLOW_TOL and nrel(x[1], y[1]) < FLOW_TOL
