"""A large grid among many small ones in one FP64 context: the launches of a workspace
group stay within the grid limits."""
import numpy as np
import pytest

from paper_1510_07799_gb300 import frg

pytestmark = pytest.mark.gpu


def test_largest_grid_in_a_full_group():
    big = frg.Params(U=1.5, T=0.64 / 256, eps_d=-0.75, N_f=256)
    small = [frg.Params(U=1.0, T=0.3, eps_d=-0.5 - 0.001 * i, N_f=2) for i in range(511)]
    mask = frg.CH_ALL | frg.NO_REVERSAL
    with frg.Context([big] + small, channel_mask=mask) as c:
        c.advance(1)
        g, s = (x.cpu().numpy() for x in c.get_state(0)[:2])
        ends = [[x.cpu().numpy() for x in c.get_state(i)[:2]] for i in (1, 511)]
    with frg.Context([big], channel_mask=mask) as c:
        c.advance(1)
        ref = [x.cpu().numpy() for x in c.get_state(0)[:2]]
    assert np.array_equal(g, ref[0]) and np.array_equal(s, ref[1])
    for p, e in zip((small[0], small[510]), ends):
        with frg.Context([p], channel_mask=mask) as c:
            c.advance(1)
            ref = [x.cpu().numpy() for x in c.get_state(0)[:2]]
        assert np.array_equal(e[0], ref[0]) and np.array_equal(e[1], ref[1])
