"""sur_lattice_step (forward, loss, gradient and Adam update of the lattice table)
against the definition in float64: classes without, with a few and with more
than 32 pairs, profile and table lengths over the staged 128 rows, samples over
the 128-wide tiles, lags of zero and more, pairs off the table, both error
normalisations; argument checks."""
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


@pytest.mark.parametrize("relative", [False, True])
@pytest.mark.parametrize("B,K,NR,m_hi,T,S,J", [(1, 1, 1, 0, 1, 0, 0), (3, 5, 2, 4, 50, 3, 2), (33, 31, 1, 9, 128, 4, 4),
                                               (70, 64, 40, 20, 129, 4, 4), (150, 140, 3, 150, 300, 4, 4),
                                               (120, 60, 3, 30, 257, 1, 5)])
def test_step_matches_definition(env, relative, B, K, NR, m_hi, T, S, J):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(B + K + T)
    f = lambda *s: torch.randn(*s, generator=g, device="cuda")
    D, moff = m_hi + K, K - 1
    G, m, v = f(NR, D, T), 1e-3 * f(NR, D, T), 1e-4 * torch.rand(NR, D, T, generator=g, device="cuda") + 1e-6
    q = -torch.rand(B, K, generator=g, device="cuda") * (torch.rand(B, K, generator=g, device="cuda") < 0.8) * 1e-9
    ant = torch.stack([torch.randint(0, NR, (B,), generator=g, device="cuda"),
                       torch.randint(0, m_hi + 1, (B,), generator=g, device="cuda")], 1).int().contiguous()
    if B > 30:
        ant[4, 0], ant[5, 0], ant[6, 1], ant[7, 1] = NR, -1, -(1 << 30), m_hi + 3 * K   # off the table
        ant[8, 1] = m_hi + 2        # meets the table's last rows only
    c_out, lr, b1, b2, eps, t = 3e9, 1e-2, 0.9, 0.999, 1e-8, 7
    trace = c_out * 1e-9 * f(B, T)
    qn, s, tn, st = torch.empty_like(q), torch.empty(B, device="cuda"), torch.empty_like(trace), torch.empty(B, device="cuda")
    fd.check(fd.sur_normalize_rows(_p(q), B, K, _p(qn), _p(s), None))
    fd.check(fd.sur_normalize_rows(_p(trace), B, T, _p(tn), _p(st), None))
    # the definition
    G64, y = G.double(), torch.zeros(B, T, dtype=torch.float64, device="cuda")
    tt = torch.arange(T, device="cuda")
    taps = []
    for b in range(B):
        ir, mb = int(ant[b, 0]), int(ant[b, 1])
        for k in range(K):
            d, tau = mb - k + moff, tt - S * k + J
            ok = (tau >= 0) & (tau < T)
            if 0 <= ir < NR and 0 <= d < D and float(qn[b, k]) != 0.0:
                taps.append((b, k, ir, d, tau[ok], tt[ok]))
                y[b, tt[ok]] += qn[b, k].double() * G64[ir, d, tau[ok]]
    s64, st64 = s.double()[:, None], st.double()[:, None]
    back = torch.ones_like(s64)
    if relative:
        back = c_out * s64 / st64
        err = y * back - tn.double()
    else:
        err = y - torch.where(s64 > 0, trace.double() / (c_out * s64), torch.zeros_like(y))
    loss, dy = (err ** 2).mean(), 2 * err / (B * T) * back
    dG = torch.zeros_like(G64)
    for b, k, ir, d, tau, at in taps:
        dG[ir, d, tau] += qn[b, k].double() * dy[b, at]
    m64 = b1 * m.double() + (1 - b1) * dG
    v64 = b2 * v.double() + (1 - b2) * dG ** 2
    W64 = G64 - lr * (m64 / (1 - b1 ** t)) / (torch.sqrt(v64 / (1 - b2 ** t)) + eps)
    # the step
    dGo, dyo, lo = torch.full_like(G, 9.0), torch.full_like(trace, 9.0), torch.full((1,), 9.0, device="cuda")
    n = fd.sur_lattice_step_bytes(B, NR)
    work = torch.empty(n, dtype=torch.uint8, device="cuda")
    args = [_p(G), _p(dGo), _p(m), _p(v), _p(qn), _p(s), _p(ant), _p(tn if relative else trace),
            _p(st) if relative else None, B, K, NR, D, T, S, J, moff, c_out, lr, b1, b2, eps, t, _p(dyo), _p(lo),
            _p(work), n, None]
    fd.check(fd.sur_lattice_step(*args))

    # float32: sums of up to K (forward) and B K / NR (gradient) products
    def close(a, r, tol):
        assert float((a.double() - r).norm()) <= tol * float(r.norm()) + 1e-30

    close(lo, loss.view(1), 2e-6)
    close(dyo, dy, 2e-6)
    close(dGo, dG, 4e-6)
    close(m, m64, 2e-6)
    close(v, v64, 2e-6)
    close(G, W64, 1e-6)
    bad = list(args); bad[26] = n - 1
    assert fd.sur_lattice_step(*bad) == -1
    bad = list(args); bad[22] = 0
    assert fd.sur_lattice_step(*bad) == -1
    assert fd.sur_lattice_step_bytes(0, 1) < 0
