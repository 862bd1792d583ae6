"""The sliced FP64 products where their integer sums or their fixed-point grids could
lose digits: lines whose digits all add up with the same sign, and lines graded along
the contraction index in opposite directions.

Reference: the direct channel's sum of one entry in extended precision.  Its error is
measured in the entry's own terms, sum |L_k| |R_k|: a bubble weight carries some ten
roundings (propagators, products, the factor T Lambda) and the sum a few more, each
2^-53 = 1.1e-16 of a term, and the terms' roundings add up at most linearly: 5e-15."""
import numpy as np
import pytest

from paper_1510_07799_gb300 import frg, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LAM = 4.0  # above the frequency box: the interaction-flow weights vary little
TOL = 5e-15


def params(N):
    # (T Lambda a power of two: the weights' factor moves no digit)
    return frg.Params(U=1.0, T=2.0 ** -np.ceil(np.log2(N)), eps_d=-0.3, N_f=N, Lambda0=1e12, Lambda_f=1.0, cutoff=1)


def propagators(p):
    """G and S of the interaction-flow cutoff at zero self-energy, extended precision."""
    ld = np.longdouble
    w = (2 * (np.arange(p.N_f) - p.N_f // 2) + 1).astype(ld) * (4 * np.arctan(ld(1))) * ld(p.T)
    gi = np.empty(p.N_f, np.clongdouble)
    gi.real, gi.imag = -(ld(p.eps_d) + ld(p.U) / 2), w + np.sign(w) * ld(p.Delta)
    G = 1 / (np.sqrt(ld(LAM)) * gi)
    return G, -G * G * gi / (2 * np.sqrt(ld(LAM)))


def direct_entry(p, V, k1, k2):
    """The direct channel's terms of the entry (k1, k2, k1), transfer 0."""
    G, S = propagators(p)
    L = 2 * S * G * np.longdouble(LAM) * np.longdouble(p.T)
    V = V.astype(np.clongdouble)
    k = np.arange(p.N_f)
    A, C = V[k1, k, k1], V[k1, k, k]
    return np.concatenate([L * (2 * A - C) * V[k, k2, k], -L * A * V[k, k2, k2]])


def direct_rhs(p, V):
    g = torch.from_numpy(V).cuda()
    s = torch.zeros(p.N_f, dtype=torch.complex128, device="cuda")
    dg, ds = torch.empty_like(g), torch.empty_like(s)
    with frg.Context([p], channel_mask=frg.CH_DPH) as c:
        c.rhs(0, LAM, g, s, dg, ds)
        c.stats()
    return dg.cpu().numpy()


def weights(p):
    G, S = propagators(p)
    return 2 * S * G


def entry_error(p, V, k1, k2):
    t = direct_entry(p, V, k1, k2)
    return float(abs(direct_rhs(p, V)[k1, k2, k1] - t.sum()) / np.abs(t).sum())


def near_top(rng, n):
    """Values whose base-256 digits all lie near 127: their products have one sign."""
    d = rng.integers(112, 128, (n, 7)).astype(np.float64)
    d[:, 0] = 126
    return (d * 256.0 ** -np.arange(7)).sum(1) / 128


@pytest.mark.parametrize("N", [28, 64, 96, 128, 160, 256])
def test_digits_that_add_up(N):
    p, rng = params(N), np.random.default_rng(N)
    V = 0.5 * inputs.random_vertex(N, p.U, seed=N, crossing=False)
    k, k1, k2 = np.arange(N), N // 3, N // 2 + 1
    # column k2: B = y (1 - i), D = -y (1 - i); row k1: (2A - C) L = 2 x (1 + i)
    V[k, k2, k] = near_top(rng, N) * (1 - 1j)
    V[k, k2, k2] = -near_top(rng, N) * (1 - 1j)
    V[k1, k, k] = 0.0
    V[k1, k, k1] = (near_top(rng, N) * (1 + 1j) / weights(p)).astype(np.complex128)
    V[k1, k2, k1] = 0.5  # (in both lines)
    assert entry_error(p, V, k1, k2) < TOL


@pytest.mark.parametrize("N", [28, 64, 130])
@pytest.mark.parametrize("decades", [1, 3, 6, 9, 30])
def test_lines_graded_in_opposite_directions(N, decades):
    """Every term of the sum is small although both lines reach one."""
    p, rng = params(N), np.random.default_rng(N)
    V = 0.5 * inputs.random_vertex(N, p.U, seed=N, crossing=False)
    k, k1, k2 = np.arange(N), N // 3, N // 2 + 1

    def z():
        return np.exp(2j * np.pi * rng.random(N)) * rng.uniform(0.5, 1.0, N)

    down, up = 10.0 ** (-decades * k / (N - 1)), 10.0 ** (-decades * (1 - k / (N - 1)))
    V[k, k2, k] = up * z()
    V[k, k2, k2] = up * z()
    V[k1, k, k] = down * z()
    V[k1, k, k1] = (down * z() / weights(p)).astype(np.complex128)
    assert entry_error(p, V, k1, k2) < TOL


@pytest.mark.parametrize("N", [28, 66])
def test_one_entry_far_above_its_line(N):
    """Per entry over the whole vertex: one value of a row and one of a column twelve
    decades above the rest, each meeting small values on the other side."""
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=N, crossing=False)
    k1, k2, a, b = N // 3, N // 2 + 1, 3, N - 4
    V[k1, a, k1] *= 1e12
    V[b, k2, b] *= 1e12
    V[b, k2, k2] *= 1e12
    got = direct_rhs(p, V)
    for q in range(N):
        for i1, i2 in ((k1, q), (q, k2), (q, (q * 7 + 3) % N)):
            t = direct_entry(p, V, i1, i2)
            assert float(abs(got[i1, i2, i1] - t.sum()) / np.abs(t).sum()) < TOL


@pytest.mark.parametrize("mask", [frg.CH_PP, frg.CH_DPH, frg.CH_XPH])
@pytest.mark.parametrize("N", [28, 66, 130])
def test_vertex_beyond_the_fixed_points(N, mask):
    """Whole tiles summed in FP64: the rhs of a vertex times 2^420 is 2^840 times the
    vertex's own (without frequencies outside the box, so U = 0).  Both sums round at
    most 8 N times, each by 2^-53 of their terms' size: 1e-12 normwise."""
    p = frg.Params(U=0.0, T=0.64 / N, eps_d=-0.3, N_f=N)
    g = torch.from_numpy(inputs.random_vertex(N, 1.3, seed=N, crossing=False)).cuda()
    s = torch.from_numpy(inputs.random_sigma(N, seed=N)).cuda()
    out = []
    with frg.Context([p], channel_mask=mask) as c:
        for e in (0, 420):
            dg, ds = torch.empty_like(g), torch.empty_like(s)
            c.rhs(0, 0.3, g * 2.0 ** e, s, dg, ds)
            out.append((dg * 2.0 ** -e * 2.0 ** -e).cpu().numpy())
        c.stats()
    assert np.max(np.abs(out[1] - out[0])) < 1e-12 * np.max(np.abs(out[0]))


@pytest.mark.parametrize("mask", [frg.CH_PP, frg.CH_DPH, frg.CH_XPH])
@pytest.mark.parametrize("N", [30, 98])
def test_one_value_that_cannot_be_sliced(N, mask):
    """Only the lines that hold it are summed in FP64; every entry as the oracle has it."""
    import oracle

    p = frg.Params(U=1.3, T=0.64 / N, eps_d=-0.3, N_f=N)
    V = inputs.random_vertex(N, p.U, seed=N, crossing=False)
    V[N // 3, N // 2, 7] = 1e150
    sig = inputs.random_sigma(N, seed=N)
    g, s = torch.from_numpy(V).cuda(), torch.from_numpy(sig).cuda()
    dg, ds = torch.empty_like(g), torch.empty_like(s)
    with frg.Context([p], channel_mask=mask) as c:
        c.rhs(0, 0.3, g, s, dg, ds)
        c.stats()
    m = oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N)
    ref, _ = oracle.rhs(m, 0.3, V, sig, mask=mask)
    huge = np.abs(ref) > 1e100
    a, b = dg.cpu().numpy(), ref
    assert huge.any() and not huge.all()
    assert np.max(np.abs(a - b)[huge] / np.abs(b)[huge]) < 1e-12
    assert np.max(np.abs(a - b)[~huge]) < 1e-12 * np.max(np.abs(b)[~huge])
