"""The FP64 flows' error norm over the whole range of FP64.  A model with every energy
(U, T, Delta, the level, the scales, the absolute tolerance) multiplied by a power of
two has the same flow, multiplied by it; only ln Lambda rounds differently, by 2^-53 of
up to 90, which a flow of some 70 attempts keeps far below 1e-8.  Steps are chosen by
the error norm, so a norm that misjudged an entry would take other steps."""
import numpy as np
import pytest

from paper_1510_07799_gb300 import frg

pytestmark = pytest.mark.gpu


def flow(N, e, mask):
    s = 2.0 ** e
    p = frg.Params(U=2.0 * s, T=0.64 / N * s, eps_d=-0.7 * s, N_f=N, Delta=s, Lambda0=1e3 * s, Lambda_f=1e-3 * s,
                   atol=1e-8 * s)
    with frg.Context([p], channel_mask=mask) as c:
        st = c.flow()[0]
        g, sig, _, _ = c.get_state(0)
    return st, g.cpu().numpy() / s, sig.cpu().numpy() / s


@pytest.mark.parametrize("N,mask", [(16, frg.CH_ALL), (16, frg.CH_ALL | frg.NO_REVERSAL), (28, frg.CH_ALL)])
@pytest.mark.parametrize("e", [130, 126, -90, -105, -115, -125])
def test_scaled_model_takes_the_same_steps(N, e, mask):
    ref, g0, s0 = flow(N, 0, mask)
    st, g, s = flow(N, e, mask)
    assert (st.accepted, st.rejected) == (ref.accepted, ref.rejected)
    assert np.max(np.abs(g - g0)) < 1e-8 * np.max(np.abs(g0))
    assert np.max(np.abs(s - s0)) < 1e-8 * np.max(np.abs(s0))
