"""The tensor-core chains lose nothing against the FP32 fast transform: W t of vectors whose
dimensions fall, rise or are alike in size, from the force rows of single atoms with sines of one."""
import numpy as np
import pytest
import torch

from oracle import sorf as o_sorf
from paper_2206_01580_gb300 import synth

pytestmark = pytest.mark.gpu

D, NF, N = 128, 1024, 999


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr
    qmlr.lib()
    return qmlr


J = np.arange(D)
SIZES = {"falling": np.exp(-J / 8.0), "falling slowly": 1.0 / (1.0 + J), "alike": np.ones(D),
         "rising": np.exp((J - 127) / 8.0), "rising slowly": 1.0 / (D - J)}


def _errors(q, t, T, sigma):
    """(mean signed relative error, relative error) of W t: tensor cores, fast transform."""
    rng = np.random.default_rng(T)
    signs, _ = synth.sorf_draw(rng, NF, D, T)
    exact = torch.as_tensor(t.astype(np.float64) @ o_sorf.sorf_matrix(signs, sigma).T).cuda()
    n = len(t) // 3
    ptr = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    words, tc_sin = q.pack_signs(signs), torch.ones((NF // D, n, D), device="cuda")
    tc = q.force_rows_tc(t, 3 * ptr.long(), ptr, tc_sin, q.sorf_tc_tables(words, T, NF), T, sigma)
    fast = q.force_rows(torch.as_tensor(t).cuda(), 3 * ptr.long(), ptr, torch.ones((n, D, NF // D), device="cuda"), words,
                        T, NF, sigma)
    assert q.device_status() == 0
    out = []
    for got in (tc, fast):
        off = got.double() - exact
        out.append((float((off * exact).sum() / exact.square().sum()), float(off.norm() / exact.norm())))
    return out


@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("T,sigma", [(3, 2.0), (2, 2.0), (3, 1.7)])
def test_error_is_not_above_the_fast_transform(q, sizes, T, sigma):
    t = (np.random.default_rng(1).normal(size=(N, D)) * SIZES[sizes]).astype(np.float32)
    (_, tc), (_, fast) = _errors(q, t, T, sigma)
    assert tc <= fast, (tc, fast)


@pytest.mark.parametrize("sizes", ["falling", "falling slowly"])
@pytest.mark.parametrize("T,sigma", [(1, 2.0), (2, 2.0), (3, 2.0), (3, 1.7)])
def test_truncations_leave_no_bias(q, sizes, T, sigma):
    """Sizes as projections on principal components have them. One truncating add at full size takes 2^-24 * 2/3
    = 4.0e-8 of a value on average; half of that is allowed (the mean over a million values is exact to ~1e-10)."""
    t = (np.random.default_rng(2).normal(size=(N, D)) * SIZES[sizes]).astype(np.float32)
    (bias, _), _ = _errors(q, t, T, sigma)
    assert abs(bias) <= 2.0e-8, bias


@pytest.mark.parametrize("power", [-100, 85, 100, 115])
def test_rows_of_any_size(q, power):
    """Vectors times a power of two give the rows times it, bit for bit: the largest of N x D normal values is below
    2^3, so |t| < 2^7 and |W t| <= sqrt(D) / sigma |t| < 2^10 at power 0, finite at 2^115."""
    signs, _ = synth.sorf_draw(np.random.default_rng(0), NF, D, 3)
    t = np.random.default_rng(3).normal(size=(N, D)).astype(np.float32)
    n = N // 3
    ptr = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    args = (3 * ptr.long(), ptr, torch.ones((NF // D, n, D), device="cuda"),
            q.sorf_tc_tables(q.pack_signs(signs), 3, NF), 3, 2.0)
    want = q.force_rows_tc(t, *args)
    got = q.force_rows_tc(np.ldexp(t, power).astype(np.float32), *args)
    assert bool(torch.isfinite(got).all()) and torch.equal(got, torch.ldexp(want, torch.tensor(power, device="cuda")))
    assert q.device_status() == 0
