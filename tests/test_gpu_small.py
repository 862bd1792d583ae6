"""FP64 right-hand sides of small grids in one launch (contexts with N_f < 24, the
allocation-free entry point up to N_f = 64), where the rows per block and the
lanes per entry change, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1510_07799_gb300 import frg, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12  # the FP64 path's bar


def nrel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def run(call, V, sig):
    g, s = torch.from_numpy(V).cuda(), torch.from_numpy(sig).cuda()
    dg, ds = torch.full_like(g, complex(np.nan, np.nan)), torch.full_like(s, complex(np.nan, np.nan))
    call(g, s, dg, ds)
    torch.cuda.synchronize()
    return dg.cpu().numpy(), ds.cpu().numpy()


@pytest.mark.parametrize("mask", [0xF, 0x9, 0x2, 0x4, 0x8])
@pytest.mark.parametrize("N", [2, 4, 8, 12, 14, 16, 18, 20, 22, 24, 26, 28, 30, 32, 34, 36, 38, 40, 42, 48, 50, 64])
def test_one_launch_rhs_matches_oracle(N, mask):
    p = frg.Params(U=1.3, T=0.64 / N, eps_d=-0.4, N_f=N)
    V = inputs.random_vertex(N, p.U, seed=N + 7 * mask, crossing=False)
    sig = inputs.random_sigma(N, seed=N)
    rg, rs = oracle.rhs(oracle.Model(U=p.U, T=p.T, eps_d=p.eps_d, Delta=p.Delta, N=N), 0.25, V, sig, mask=mask)
    got = [run(lambda *a: frg.rhs_noalloc(p, 0.25, *a, channel_mask=mask), V, sig)]
    with frg.Context([p], channel_mask=mask) as ctx:
        got.append(run(lambda *a: ctx.rhs(0, 0.25, *a), V, sig))
    for dg, ds in got:
        assert nrel(dg, rg) < TOL if mask & 7 else np.max(np.abs(dg)) == 0.0
        assert nrel(ds, rs) < TOL if mask & 8 else np.max(np.abs(ds)) == 0.0


def test_batch_of_small_and_sliced_points():
    """Each point of a mixed context gets bitwise the rhs of its own context."""
    pts = [frg.Params(U=1.0 + 0.2 * i, T=0.64 / n, eps_d=-0.3, N_f=n) for i, n in enumerate((2, 22, 24, 16, 40))]
    with frg.Context(pts) as ctx:
        ctx.advance(2)
        both = [ctx.get_state(i)[:2] for i in range(len(pts))]
    for p, (g, s) in zip(pts, both):
        with frg.Context([p]) as one:
            one.advance(2)
            g1, s1, _, _ = one.get_state(0)
        assert torch.equal(g, g1) and torch.equal(s, s1)


@pytest.mark.parametrize("N", [16, 64])
def test_self_energy_rhs_in_place(N):
    """The self-energy output may be the input's own buffer."""
    p = frg.Params(U=1.3, T=0.64 / N, eps_d=-0.4, N_f=N)
    V = torch.from_numpy(inputs.random_vertex(N, p.U, seed=N)).cuda()
    sig = torch.from_numpy(inputs.random_sigma(N, seed=N)).cuda()
    calls = [lambda *a: frg.rhs_noalloc(p, 0.25, *a)]
    with frg.Context([p]) as ctx, frg.Context([p], precision="3xtf32") as split, \
            frg.Context([p], precision="bf16x3", channel_mask=frg.CH_ALL | frg.TAILS) as tails:
        calls += [lambda *a, c=c: c.rhs(0, 0.25, *a) for c in (ctx, split, tails)]
        for call in calls:
            dg, ds, dg2, buf = torch.empty_like(V), torch.empty_like(sig), torch.empty_like(V), sig.clone()
            call(V, sig, dg, ds)
            call(V, buf, dg2, buf)
            torch.cuda.synchronize()
            assert torch.equal(dg, dg2) and torch.equal(ds, buf)


def test_threads_with_different_sizes():
    """Calls of different sizes from several threads, each on a stream of its own."""
    import threading

    cases, errors = [], []
    for N in (36, 48, 56, 64):
        p = frg.Params(U=1.3, T=0.64 / N, eps_d=-0.4, N_f=N)
        V = torch.from_numpy(inputs.random_vertex(N, p.U, seed=N)).cuda()
        sig = torch.from_numpy(inputs.random_sigma(N, seed=N)).cuda()
        ref = torch.empty_like(V), torch.empty_like(sig)
        frg.rhs_noalloc(p, 0.25, V, sig, *ref)
        cases.append((p, V, sig, ref, (torch.empty_like(V), torch.empty_like(sig)), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def work(p, V, sig, ref, out, stream):
        try:
            with torch.cuda.stream(stream):
                for _ in range(200):
                    frg.rhs_noalloc(p, 0.25, V, sig, *out)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=c) for c in cases]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for c in cases:
        assert torch.equal(c[3][0], c[4][0]) and torch.equal(c[3][1], c[4][1])
