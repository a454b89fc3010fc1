"""The solve and the exact operator with a workspace of one partial sum per 2048 rows: the bits of
the larger workspace, and a smaller one refused."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr
    qmlr.lib()
    return qmlr


def _saved(n_rows, n):
    """Bytes between one sum per 128 rows and one per 2048."""
    folds = max(-(-n_rows // 128), 1)
    return (folds - max(-(-n_rows // 2048), 1)) * n * 8


def _call(q, f, need, *args):
    """f with `need` bytes of 256-byte aligned workspace, in front of bytes that must stay."""
    buf = torch.full((need + 512,), 0x5A, device="cuda", dtype=torch.uint8)
    at = buf.data_ptr() + (-buf.data_ptr()) % 256
    rc = f(*args, at, need, q._stream())
    torch.cuda.synchronize()
    end = at - buf.data_ptr() + need
    assert bool((buf[end:] == 0x5A).all())
    return rc


@pytest.mark.parametrize("n_rows,n", [(0, 8), (1, 4), (128, 64), (2047, 7), (2049, 1024), (6000, 516), (33000, 130)])
def test_operator_with_the_small_workspace(q, n_rows, n):
    g = torch.Generator(device="cuda").manual_seed(n_rows)
    Z = torch.randn((n_rows, n), device="cuda", generator=g)
    p = torch.randn(n, device="cuda", generator=g, dtype=torch.float64)
    want = q.normal_apply(Z, p, 0.5)
    need = q.lib().qmlr_normal_apply_workspace_bytes(n_rows, n) - _saved(n_rows, n)
    out = torch.zeros_like(p)
    args = (q._ptr(Z) if n_rows else None, n_rows, n, n, 0.5, q._ptr(p), q._ptr(out))
    assert _call(q, q.lib().qmlr_normal_apply, need, *args) == q.OK
    assert torch.equal(out, want)
    assert _call(q, q.lib().qmlr_normal_apply, need - 1, *args) == q.EINVAL


@pytest.mark.parametrize("n_rows,n", [(300, 64), (5000, 512)])
def test_solve_with_the_small_workspace(q, n_rows, n):
    import ctypes as C
    g = torch.Generator(device="cuda").manual_seed(n)
    Z = torch.randn((n_rows, n), device="cuda", generator=g)
    y = torch.randn(n_rows, device="cuda", generator=g, dtype=torch.float64)
    G = q.gram(Z, q.GRAM_FP32)
    want, it, _ = q.gram_solve(G, Z, y, 1e-3)
    need = q.lib().qmlr_solve_workspace_bytes(n_rows, n) - _saved(n_rows, n)
    alpha = torch.zeros(n, device="cuda", dtype=torch.float64)
    opts = q.SolveOpts(q.SOLVE_PCG, 50, 1e-10, -2.0 ** -16, 0, 0.0, 0.0, 0.0, 0.0, q.FACTOR_MIXED)
    args = (q._ptr(G), q._ptr(Z), n_rows, n, n, q._ptr(y), 1e-3, C.byref(opts), q._ptr(alpha))
    assert _call(q, q.lib().qmlr_gram_solve, need, *args) == q.OK
    assert torch.equal(alpha, want) and opts.iters_done == it
    assert _call(q, q.lib().qmlr_gram_solve, need - 1, *args) == q.EINVAL
    assert q.device_status() == 0
