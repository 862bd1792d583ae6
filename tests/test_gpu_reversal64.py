"""FP64 flows under the frequency-reversal reduction: the transfers m < N and the
entries i1 < N/2 formed, the others as conjugates of their mirrors.

The sliced products are exact integer sums, the other sums are formed for the entry
itself: per rhs the reduction changes an entry by the rounding of its mirror's sum
(an N-term FP64 sum: 2 N 2^-53 of its terms' size; 40 attempts of seven such sums
and a factor 10 for the flow's amplification give 1e-11 at N = 130 normwise), at
the same scale: the step control divides differences of rounding size by the error
norm, so that two flows may stand some 1e-10 apart in ln Lambda after equally many
attempts, and one state is moved to the other's scale along its rhs before they are
compared."""
import numpy as np
import pytest
import torch

from paper_1510_07799_gb300 import frg, inputs

pytestmark = pytest.mark.gpu
TOL = 1e-11


def params(N, asym=0.3):
    return frg.Params(U=1.5, T=0.64 / N, eps_d=-0.75 + asym, N_f=N)


def run(pts, mask, states=None, n=6):
    with frg.Context(pts, channel_mask=mask) as c:
        if states:
            for i, (g, s, lam) in enumerate(states):
                c.set_state(i, g, s, lam)
        st = c.advance(n)
        out = []
        for i in range(len(pts)):
            g, s, lam, _ = c.get_state(i)
            dg, ds = torch.empty_like(g), torch.empty_like(s)
            c.rhs(i, lam, g, s, dg, ds)
            out.append([x.cpu().numpy() for x in (g, s)] + [np.log(lam)] + [x.cpu().numpy() for x in (dg, ds)])
        return out, [x.rhs_evals for x in st]


def nrel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def close(a, b, part):
    """Part 0 (vertex) or 1 (self-energy) of two states, the first one moved to the
    other's scale."""
    dl = b[2] - a[2]
    assert abs(dl) < 1e-8
    return nrel(a[part] + dl * a[3 + part], b[part]) < TOL


def mirrored(g, s):
    return np.conj(g.ravel()[::-1]).reshape(g.shape), np.conj(s[::-1])


@pytest.mark.parametrize("N", [2, 4, 10, 16, 18, 24, 26, 28, 30, 34, 62, 64, 66, 82, 130])
def test_reduced_flow(N):
    p = [params(N)]
    (a,), ea = run(p, frg.CH_ALL)
    (b,), eb = run(p, frg.CH_ALL | frg.NO_REVERSAL)
    assert ea == eb
    assert close(a, b, 0) and close(a, b, 1)
    for x, y in zip(a[:2], mirrored(*a[:2])):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("mask", [frg.CH_PP | frg.CH_SIGMA, frg.CH_DPH, frg.CH_XPH | frg.CH_SIGMA, frg.CH_PP | frg.CH_XPH])
@pytest.mark.parametrize("N", [14, 46])
def test_channel_subsets(N, mask):
    (a,), _ = run([params(N)], mask)
    (b,), _ = run([params(N)], mask | frg.NO_REVERSAL)
    assert close(a, b, 0)
    if mask & frg.CH_SIGMA:
        assert close(a, b, 1)


def test_mixed_grids_and_a_state_without_the_symmetry():
    """Symmetric states keep the reduction; one state without the symmetry turns it
    off for the context, bitwise the flow that computes every transfer; a symmetric
    one brings it back."""
    pts = [params(N) for N in (12, 40, 70, 24)]
    (a, _), (b, _) = run(pts, frg.CH_ALL), run(pts, frg.CH_ALL | frg.NO_REVERSAL)
    for x, y in zip(a, b):
        assert close(x, y, 0) and close(x, y, 1)
    states = []
    for p in pts:
        g = torch.from_numpy(inputs.random_vertex(p.N_f, p.U, seed=3)).cuda()
        states.append((g, torch.from_numpy(inputs.random_sigma(p.N_f, seed=4)).cuda(), 2.0))
    sym = []
    for g, s, lam in states:
        mg, ms = mirrored(g.cpu().numpy(), s.cpu().numpy())
        sym.append((torch.from_numpy(0.5 * (g.cpu().numpy() + mg)).cuda(),
                    torch.from_numpy(0.5 * (s.cpu().numpy() + ms)).cuda(), lam))
    mixed = [sym[0], states[1], sym[2], sym[3]]
    (a, _), (b, _) = run(pts, frg.CH_ALL, mixed, 3), run(pts, frg.CH_ALL | frg.NO_REVERSAL, mixed, 3)
    for x, y in zip(a, b):
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
    (a, _), (b, _) = run(pts, frg.CH_ALL, sym, 3), run(pts, frg.CH_ALL | frg.NO_REVERSAL, sym, 3)
    for x, y in zip(a, b):
        assert close(x, y, 0) and close(x, y, 1)
    with frg.Context(pts, channel_mask=frg.CH_ALL) as c:
        for st, want in ((mixed, False), (sym, True)):
            for i, (g, s, lam) in enumerate(st):
                c.set_state(i, g, s, lam)
            c.advance(3)
            ref, _ = run(pts, frg.CH_ALL, st, 3)
            for i, r in enumerate(ref):
                g, s = c.get_state(i)[:2]
                assert np.array_equal(g.cpu().numpy(), r[0]) and np.array_equal(s.cpu().numpy(), r[1])


@pytest.mark.parametrize("N", [16, 36])
def test_resumed_flow_is_the_same(N):
    """A state read and set again, with its step, continues bit for bit."""
    p = [params(N)]
    with frg.Context(p) as c:
        c.advance(4)
        g, s, lam, h = c.get_state(0)
        g, s = g.clone(), s.clone()
        c.set_state(0, g, s, lam, h)
        c.advance(3)
        a = [x.cpu().numpy() for x in c.get_state(0)[:2]]
    with frg.Context(p) as c:
        c.set_state(0, g, s, lam, h)
        c.advance(3)
        b = [x.cpu().numpy() for x in c.get_state(0)[:2]]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for x, y in zip(a, mirrored(*a)):
        assert np.array_equal(x, y)
