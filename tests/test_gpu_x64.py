"""FP64 channel products by exact slices on the tensor cores (grids with N_f >= 28)
against the oracle and against extended-precision sums, at the edges of their
tiles (64 rows and columns, 16 k), for values that cannot be sliced, and for
contexts whose operands do not fit one workspace."""
import numpy as np
import pytest

import oracle
from paper_1510_07799_gb300 import frg, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RHS_TOL = 1e-12  # the FP64 path's bar


def nrel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def params(N, U=1.7):
    return frg.Params(U=U, T=0.64 / N, eps_d=-0.5 * U + 0.3, N_f=N)


def ctx_rhs(ctx, Lam, V, sig):
    g, s = torch.from_numpy(V).cuda(), torch.from_numpy(sig).cuda()
    dg, ds = torch.full_like(g, complex(np.nan, np.nan)), torch.full_like(s, complex(np.nan, np.nan))
    ctx.rhs(0, Lam, g, s, dg, ds)
    ctx.stats()  # synchronises and reports a wait that ran out
    return dg.cpu().numpy(), ds.cpu().numpy()


def core_rhs(p, Lam, V, sig):
    """The same through the CUDA cores (the allocation-free entry point)."""
    g, s = torch.from_numpy(V).cuda(), torch.from_numpy(sig).cuda()
    dg, ds = torch.empty_like(g), torch.empty_like(s)
    frg.rhs_noalloc(p, Lam, g, s, dg, ds)
    torch.cuda.synchronize()
    return dg.cpu().numpy(), ds.cpu().numpy()


@pytest.mark.parametrize("mask", [0xF, 0x1, 0x2, 0x4, 0x6])
@pytest.mark.parametrize("N", [28, 30, 32, 48, 62, 66, 82, 96])
def test_rhs_matches_oracle_at_tile_edges(N, mask):
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=N + mask, crossing=False)
    sig = inputs.random_sigma(N, seed=N)
    with frg.Context([p], channel_mask=mask) as ctx:
        dg, _ = ctx_rhs(ctx, 0.3, V, sig)
    rg, _ = oracle.rhs(oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N), 0.3, V, sig, mask=mask)
    assert nrel(dg, rg) < RHS_TOL


@pytest.mark.parametrize("N", [126, 130, 192, 256])
def test_rhs_matches_oracle_on_large_grids(N):
    """Several row and column tiles; 400 entries, the corners among them."""
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=N, crossing=False)
    sig = inputs.random_sigma(N, seed=N)
    with frg.Context([p]) as ctx:
        dg, _ = ctx_rhs(ctx, 0.1, V, sig)
    idx = np.random.default_rng(N).integers(0, N, (400, 3))
    idx[:8] = [[a, b, c] for a in (0, N - 1) for b in (0, N - 1) for c in (0, N - 1)]
    ref = oracle.rhs_entries(oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N), 0.1, V, sig, idx)
    assert nrel(dg[idx[:, 0], idx[:, 1], idx[:, 2]], ref) < RHS_TOL


def extended_rhs(p, Lam, V, sig, idx):
    """The channel sums of the entries idx in extended precision (numpy's long
    double: 64 or more significant bits)."""
    N, ld = p.N_f, np.longdouble
    k = np.arange(N)
    w = (2 * (k - N // 2) + 1).astype(ld) * (4 * np.arctan(ld(1))) * ld(p.T)
    th, dth = 1 + ld(Lam) ** 2 / w ** 2, 2 * ld(Lam) / w ** 2
    gi = np.empty(N, np.clongdouble)
    gi.real, gi.imag = -(ld(p.eps_d) + ld(p.U) / 2), w + np.sign(w) * ld(p.Delta)
    G = 1 / (th * gi - sig)
    S = -dth * G * G * gi

    def at(i1, i2, i3):
        i1, i2, i3 = np.broadcast_arrays(i1, i2, i3)
        i4 = i1 + i2 - i3
        ok = (np.minimum.reduce([i1, i2, i3, i4]) >= 0) & (np.maximum.reduce([i1, i2, i3, i4]) < N)
        c = [np.clip(i, 0, N - 1) for i in (i1, i2, i3)]
        return np.where(ok, V[c[0], c[1], c[2]], p.U).astype(np.clongdouble)

    def bub(a, b):
        c = np.clip(b, 0, N - 1)
        return np.where((b >= 0) & (b < N), S[a] * G[c] + G[a] * S[c], 0)

    out = []
    for k1, k2, k3 in idx:
        s, t, q, k4 = k1 + k2, k3 - k1, k2 - k3, k1 + k2 - k3
        pp = -(at(k1, k2, k) * bub(k, s - k) * at(k, s - k, k3)).sum()
        A, D = at(k1, k, k3), at(k - t, k2, k)
        L = bub(k, k - t)
        dd = (L * (2 * A * D - at(k1, k, k - t) * D - A * at(k - t, k2, k4))).sum()
        xx = -(at(k1, k + q, k) * bub(k, k + q) * at(k, k2, k3)).sum()
        out.append((pp + dd + xx) * ld(Lam) * ld(p.T))
    return np.array(out)


@pytest.mark.parametrize("N", [28, 48, 64])
@pytest.mark.parametrize("Lam", [0.02, 0.2])
@pytest.mark.parametrize("spread", [0.0, 3.0])
def test_error_is_no_larger_than_the_cuda_cores(N, Lam, spread):
    """Root-mean-square error against extended precision, also for vertices
    whose entries spread over decades.  The sliced sum rounds once, the chain
    of fused multiply-adds at every term; both carry the rounding of the bubble
    weights, hence the margin of a quarter."""
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=5 + N, crossing=False)
    if spread:
        V = V * 10.0 ** np.random.default_rng(N).uniform(-spread, 0.0, V.shape)
    sig = inputs.random_sigma(N, seed=6)
    idx = np.random.default_rng(7).integers(0, N, (1500, 3))
    ref = extended_rhs(p, Lam, V, sig, idx)
    at = (idx[:, 0], idx[:, 1], idx[:, 2])
    with frg.Context([p]) as ctx:
        sliced = ctx_rhs(ctx, Lam, V, sig)[0][at]
    core = core_rhs(p, Lam, V, sig)[0][at]
    rms = [float(np.sqrt(np.mean(np.abs(x - ref) ** 2) / np.mean(np.abs(ref) ** 2))) for x in (sliced, core)]
    assert rms[0] <= 1.25 * rms[1] and rms[0] < 2e-15, rms


@pytest.mark.parametrize("what", ["nan", "inf", "huge", "tiny", "zero"])
def test_values_that_cannot_be_sliced(what):
    """Non-finite and extreme values give what the CUDA cores give, and the next
    evaluation of the context is unaffected."""
    N = 34
    p = params(N)
    V0 = inputs.random_vertex(N, p.U, seed=3, crossing=False)
    sig = inputs.random_sigma(N, seed=4)
    V = V0.copy()
    if what in ("nan", "inf"):
        V[5, 20, 9] = complex(np.nan if what == "nan" else np.inf, 0.5)
    elif what == "zero":
        V[:] = 0.0
    else:
        V *= 1e140 if what == "huge" else 1e-140
    with frg.Context([p]) as ctx:
        base, _ = ctx_rhs(ctx, 0.4, V0, sig)
        got, _ = ctx_rhs(ctx, 0.4, V, sig)
        again, _ = ctx_rhs(ctx, 0.4, V0, sig)
    want, _ = core_rhs(p, 0.4, V, sig)
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        fine = np.isfinite(b)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isfinite(a), fine)
        assert np.array_equal(a[~fine & ~np.isnan(b)], b[~fine & ~np.isnan(b)])
        scale = max(float(np.max(np.abs(b[fine]))), 1e-300)
        assert float(np.max(np.abs(a[fine] / scale - b[fine] / scale))) < RHS_TOL
    assert np.array_equal(base, again)


def test_points_in_several_workspace_groups():
    """Fourteen N = 128 points need more than one workspace; each point's step is
    bitwise that of a context holding it alone, next to points on the CUDA cores."""
    pts = [params(128, U=1.0 + 0.1 * i) for i in range(14)] + [params(8), params(40)]
    with frg.Context(pts) as ctx:
        ctx.advance(1)
        batched = [ctx.get_state(i)[:2] for i in (0, 13, 14, 15)]
    for i, (g, s) in zip((0, 13, 14, 15), batched):
        with frg.Context([pts[i]]) as one:
            one.advance(1)
            g1, s1, _, _ = one.get_state(0)
        assert torch.equal(g, g1) and torch.equal(s, s1)


def test_tails_with_sliced_products():
    N = 40
    p = params(N)
    V = inputs.random_vertex(N, p.U, seed=8, crossing=False)
    sig = inputs.random_sigma(N, seed=9)
    m = oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N)
    with frg.Context([p], channel_mask=frg.CH_ALL | frg.TAILS) as ctx:
        dg, ds = ctx_rhs(ctx, 0.3, V, sig)
    rg, rs = oracle.rhs(m, 0.3, V, sig, mask=frg.CH_ALL | frg.TAILS)
    assert nrel(dg, rg) < RHS_TOL and nrel(ds, rs) < RHS_TOL
