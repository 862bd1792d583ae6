"""Split flows whose stage kernels take narrow blocks (several points, or a grid whose
blocks do not fit the SMs in one go) against the same points alone (wide blocks): the
block shape changes no arithmetic, so the states agree bit for bit."""
import pytest
import torch

from paper_1510_07799_gb300 import frg

pytestmark = pytest.mark.gpu


def point(N, i):
    return frg.Params(U=1.0 + 0.2 * i, T=0.64 / N, eps_d=-0.4 - 0.1 * i, N_f=N)


def states(pts, precision, mask):
    with frg.Context(pts, precision=precision, channel_mask=mask) as c:
        st = c.advance(3)
        return [c.get_state(i)[:2] for i in range(len(pts))], [s.rhs_evals for s in st]


@pytest.mark.parametrize("sizes", [(128, 98), (66, 2, 34, 64, 100, 10, 80, 128)])
@pytest.mark.parametrize("precision,extra", [("3xtf32", 0), ("bf16x3", 0), ("3xtf32", frg.NO_REVERSAL),
                                             ("bf16x3", frg.TAILS), ("3xtf32", frg.REVERSAL)])
def test_narrow_blocks_give_the_wide_blocks_states(sizes, precision, extra):
    pts = [point(N, i) for i, N in enumerate(sizes)]
    got, ev = states(pts, precision, frg.CH_ALL | extra)
    for i, p in enumerate(pts):
        (ref,), (e,) = states([p], precision, frg.CH_ALL | extra)
        assert e == ev[i]
        assert torch.equal(ref[0], got[i][0]) and torch.equal(ref[1], got[i][1])
