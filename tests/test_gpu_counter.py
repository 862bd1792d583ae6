"""The launch counter under several host threads: every launch counts once, also beside
contexts that record and replay their step graphs."""
import threading

import pytest
import torch

from paper_1510_07799_gb300 import frg, inputs

pytestmark = pytest.mark.gpu


def noalloc_calls(n):
    p = frg.Params(U=1.3, T=0.1, eps_d=-0.4, N_f=4)
    V = torch.from_numpy(inputs.random_vertex(4, p.U, seed=1)).cuda()
    s = torch.from_numpy(inputs.random_sigma(4, seed=2)).cuda()
    out = torch.empty_like(V), torch.empty_like(s)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        for _ in range(n):
            frg.rhs_noalloc(p, 0.25, V, s, *out)
    st.synchronize()


def flows(n):
    for _ in range(n):
        with frg.Context([frg.Params(U=1.0, T=0.05, eps_d=-0.5, N_f=12)]) as c:
            c.advance(2)


def counted(*work):
    n0 = frg.kernel_launches()
    threads = [threading.Thread(target=f, args=(n,)) for f, n in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return frg.kernel_launches() - n0


def test_every_launch_counts_once():
    counted((noalloc_calls, 1), (flows, 1))  # (load the library and the kernels)
    call, flow = counted((noalloc_calls, 100)) / 100, counted((flows, 1))
    assert call == 1 and flow > 0
    assert counted(*[(noalloc_calls, 2500)] * 6, (flows, 20)) == 6 * 2500 + 20 * flow
