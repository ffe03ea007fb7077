"""sur_gemm_bf16 with transposed (MN-major) operands on the tcgen05 kernels (the
split-K cluster kernel for few output tiles, the persistent one for many)
against the FP64 product of the same bf16 operands: ragged sizes, K remainders,
padded rows holding garbage, the fused epilogue, accumulation; unaligned rows
still take mma.sync; column sums and the ReLU gradient at their vector and
cluster edges."""
import ctypes as C

import numpy as np
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


def _operand(torch, g, rows, K, kmajor, pad):
    """The operand [rows, K] in float64, and its storage with a row stride that
    is a multiple of 8 (pad 0) or odd (pad 1)."""
    r, c = (rows, K) if kmajor else (K, rows)
    ld = (c + 7) // 8 * 8 + 8 + pad
    t = torch.full((r, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    t[:, :c] = torch.randn(r, c, generator=g, device="cuda").bfloat16()
    v = t[:, :c].double()
    return (v if kmajor else v.T), t, ld


@pytest.mark.parametrize("ak,bk", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (70, 50, 40), (128, 128, 64), (129, 200, 2112), (257, 130, 30),
                                   (64, 256, 8200), (1024, 96, 4096), (1500, 1600, 96), (4096, 520, 72)])
def test_transposed_operands(env, M, N, K, ak, bk):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(M + 3 * N + 7 * K)
    a, A, lda = _operand(torch, g, M, K, ak, 0)
    b, B, ldb = _operand(torch, g, N, K, bk, 0)
    bias = torch.randn(N, generator=g, device="cuda")
    ref = a @ b.T
    ldy = N + 3
    n0 = fd.sur_gemm_tc_launches()
    Y = torch.zeros(M, ldy, device="cuda")
    Yb = torch.zeros(M, ldy, dtype=torch.bfloat16, device="cuda")
    fd.check(fd.sur_gemm_bf16(_p(A), lda, ak, _p(B), ldb, bk, _p(Y), ldy, _p(Yb), M, N, K, _p(bias), 1, 0, None))
    want = (ref + bias.double()).clamp_min(0)
    tol = 2e-5 * max(1.0, float(ref.abs().max()))   # f32 accumulation of K bf16 products, as for K-major operands
    assert float((Y[:, :N].double() - want).abs().max()) <= tol
    assert torch.equal(Yb[:, :N], Y[:, :N].bfloat16()) and not Y[:, N:].any()
    fd.check(fd.sur_gemm_bf16(_p(A), lda, ak, _p(B), ldb, bk, _p(Y), ldy, None, M, N, K, None, 0, 1, None))
    assert float((Y[:, :N].double() - want - ref).abs().max()) <= 2 * tol
    assert fd.sur_gemm_tc_launches() - n0 == 2 and fd.sur_gemm_tc_failed() == 0


def test_unaligned_rows_take_mma_sync(env):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    M, N, K = 100, 90, 70
    a, A, lda = _operand(torch, g, M, K, 0, 1)
    b, B, ldb = _operand(torch, g, N, K, 0, 0)
    n0 = fd.sur_gemm_tc_launches()
    Y = torch.zeros(M, N, device="cuda")
    fd.check(fd.sur_gemm_bf16(_p(A), lda, 0, _p(B), ldb, 0, _p(Y), N, None, M, N, K, None, 0, 0, None))
    assert fd.sur_gemm_tc_launches() == n0
    assert float((Y.double() - a @ b.T).abs().max()) <= 2e-5 * float((a @ b.T).abs().max())


@pytest.mark.parametrize("M,N,pad", [(1, 1, 0), (7, 33, 1), (255, 64, 0), (256, 31, 2), (4096, 1024, 0), (9001, 70, 5)])
def test_column_sums(env, M, N, pad):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    z = torch.randn(M, N + pad, generator=g, device="cuda")
    db = torch.full((N,), 9.0, device="cuda")
    fd.check(fd.sur_bias_grad(_p(z), N + pad, M, N, _p(db), None))
    want = z[:, :N].double().sum(0)
    # float32 sums: at most M / 8 + 44 roundings of partial sums below sum |z|
    bound = 2.0 ** -24 * (M / 8 + 44) * z[:, :N].double().abs().sum(0) / 8 + 1e-30
    assert bool(((db.double() - want).abs() <= torch.maximum(bound, 1e-6 * z[:, :N].double().abs().sum(0))).all())


@pytest.mark.parametrize("n,off", [(1, 0), (3, 0), (4, 0), (4096, 0), (4096, 1), (1000003, 0)])
@pytest.mark.parametrize("with_bf16", [True, False])
def test_relu_gradient(env, n, off, with_bf16):
    torch, fd = env
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    y, dy = (torch.randn(n + off, generator=g, device="cuda")[off:] for _ in range(2))
    dz, zb = torch.zeros(n, device="cuda"), torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    fd.check(fd.sur_relu_bwd(_p(y), _p(dy), _p(dz), _p(zb) if with_bf16 else None, n, None))
    want = torch.where(y > 0, dy, torch.zeros_like(dy))
    assert torch.equal(dz, want) and (not with_bf16 or torch.equal(zb, want.bfloat16()))
