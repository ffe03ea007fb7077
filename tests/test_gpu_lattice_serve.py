"""sur_lattice_serve (every profile at every antenna) against the definition in
float64 from the same split tables: tile edges in profiles and samples, profile
lengths that are not a multiple of 64, lags that are not a multiple of four
(scalar weight copies), antennas off the table, a zero profile; argument checks."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    torch.cuda.set_device(0)
    import paper_1001_5341_gb300 as fd
    return torch, fd


def _p(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("P,A,K,T,S,J", [(1, 1, 1, 1, 4, 4), (3, 5, 31, 40, 4, 4), (64, 4, 128, 1024, 4, 4),
                                         (128, 3, 64, 500, 4, 4), (129, 2, 65, 130, 3, 2), (200, 7, 100, 257, 1, 0),
                                         (70, 300, 20, 96, 8, 8)])
def test_matches_definition(env, P, A, K, T, S, J):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(P + A + K + T)
    NR, m_hi = 5, 17
    D, moff = m_hi + K, K - 1
    G = torch.randn(NR, D, T, generator=g, device="cuda")
    hi, lo = torch.empty_like(G, dtype=torch.bfloat16), torch.empty_like(G, dtype=torch.bfloat16)
    fd.check(fd.sur_split_bf16(_p(G), _p(hi), _p(lo), G.numel(), None))
    q = -torch.rand(P, K, generator=g, device="cuda") * 1e-9
    if P > 2:
        q[1] = 0
    ant = torch.stack([torch.randint(0, NR, (A,), generator=g, device="cuda"),
                       torch.randint(0, m_hi + 1, (A,), generator=g, device="cuda")], 1).int().contiguous()
    if A > 4:
        ant[2, 0], ant[3, 1] = NR, m_hi + 5   # a class and offsets off the table contribute zeros
    n = fd.sur_lattice_serve_bytes(P, A, K, T)
    work = torch.empty(n, dtype=torch.uint8, device="cuda")
    out = torch.full((A, P, T), 9.0, device="cuda")
    args = [_p(hi), _p(lo), _p(q), _p(ant), P, A, K, NR, D, T, S, J, moff, 2.5, _p(work), n, _p(out), None]
    fd.check(fd.sur_lattice_serve(*args))
    tab = hi.double() + lo.double()
    W = torch.zeros(A, K, T, dtype=torch.float64, device="cuda")
    t = torch.arange(T, device="cuda")
    for a in range(A):
        ir, m = int(ant[a, 0]), int(ant[a, 1])
        for k in range(K):
            d, tau = m - k + moff, t - S * k + J
            ok = (tau >= 0) & (tau < T)
            if ir < NR and 0 <= d < D:
                W[a, k, ok] = tab[ir, d, tau[ok]]
    peak = q.double().abs().amax(1, keepdim=True)
    qn = torch.where(peak > 0, q.double() / peak.clamp_min(1e-300), torch.zeros_like(q.double()))
    want = 2.5 * peak * (qn @ W)
    # split operands drop lo * lo (2^-17 of each factor), f32 sums of 3 K products
    tol = 2.5 * peak * (2.0 ** -15 * qn.abs() @ W.abs() + 1e-30)
    assert bool(((out.double() - want).abs() <= tol).all())
    assert fd.sur_gemm_tc_failed() == 0
    bad = list(args); bad[15] = n - 1
    assert fd.sur_lattice_serve(*bad) == -1
    bad = list(args); bad[5] = 65536
    assert fd.sur_lattice_serve(*bad) == -1
    assert fd.sur_lattice_serve_bytes(0, 1, 1, 1) < 0
