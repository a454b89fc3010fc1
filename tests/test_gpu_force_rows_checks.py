"""qmlr_force_rows_tc with arguments that do not belong together: outputs of another layout are refused
on the host, and offsets that do not match the rows or the atoms become a device error, the rows of the
other molecules being right."""
import numpy as np
import pytest
import torch

from paper_2206_01580_gb300 import synth

D, NF, T = 128, 256, 3
BAD_INDEX = 3


@pytest.mark.parametrize("out,row0,what", [
    (torch.zeros((15, NF), dtype=torch.float64), 0, "float32"), (torch.zeros(15 * NF), 0, "float32"),
    (torch.zeros((NF, 15)).T, 0, "float32"), (torch.zeros((15, NF - 1)), 0, "columns"),
    (torch.zeros(NF).expand(15, NF), 0, "columns"), (torch.zeros((14, NF)), 0, "rows"),
    (torch.zeros((17, NF)), 3, "rows"), (torch.zeros((17, NF)), -1, "rows"), (torch.zeros((17, NF)), 2, "device")])
def test_refused_outputs(out, row0, what):
    from paper_2206_01580_gb300 import qmlr
    sin_t = torch.zeros((NF // D, 5, D))
    with pytest.raises(AssertionError, match=what):
        qmlr.force_rows_tc(torch.zeros((3, D)), torch.zeros(2, dtype=torch.int64), torch.zeros(2, dtype=torch.int32),
                           sin_t, torch.zeros(4 * NF * D, dtype=torch.int16), T, 2.0, out=out, row0=row0)


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr
    qmlr.lib()
    return qmlr


SIZES = np.array([7, 3, 1, 21])


def _inputs(q, extra_rows=0):
    rng = np.random.default_rng(4)
    mol_ptr = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int32)
    jac_ptr = np.concatenate([[0], np.cumsum(3 * SIZES.astype(np.int64) ** 2)])
    t = rng.normal(size=(int(jac_ptr[-1]) + extra_rows, D)).astype(np.float32)
    signs, _ = synth.sorf_draw(rng, NF, D, T)
    sin_t = torch.as_tensor(rng.normal(size=(NF // D, int(mol_ptr[-1]), D)).astype(np.float32)).cuda()
    return mol_ptr, jac_ptr, t, sin_t, q.sorf_tc_tables(q.pack_signs(signs), T, NF)


@pytest.mark.gpu
@pytest.mark.parametrize("case", ["more rows", "fewer rows", "short molecule", "atoms beyond", "late start"])
def test_offsets_that_do_not_match(q, case):
    mol_ptr, jac_ptr, t, sin_t, tables = _inputs(q, 130 * 3)
    want = q.force_rows_tc(t[:jac_ptr[-1]], jac_ptr, mol_ptr, sin_t, tables, T, 2.0).cpu()
    assert q.device_status() == 0
    good = [0, 1, 2, 3]
    rows = int(jac_ptr[-1])
    bad_mol, bad_jac = mol_ptr.copy(), jac_ptr.copy()
    if case == "more rows":        # tangents after the last molecule's
        rows += 130 * 3
    elif case == "fewer rows":     # the last molecule's rows end early
        rows -= 3 * 21
        good = [0, 1, 2]
    elif case == "short molecule":   # two molecules' atoms do not have these rows
        bad_mol[1] -= 1
        good = [2, 3]
    elif case == "atoms beyond":   # the last molecule has more atoms than sin_t, and rows for them
        bad_mol[-1] += 1
        bad_jac[-1] = bad_jac[-2] + 3 * 22 ** 2
        rows = int(bad_jac[-1])
        good = [0, 1, 2]
    else:
        bad_jac[0] = 3             # rows before the first molecule
        good = [1, 2, 3]
    out = torch.full((int(mol_ptr[-1]) * 3 + 9, NF), 7.0, device="cuda")
    q.force_rows_tc(t[:rows], bad_jac, bad_mol, sin_t, tables, T, 2.0, out=out, row0=4)
    torch.cuda.synchronize()
    assert q.device_status() == BAD_INDEX
    out = out.cpu()
    assert bool((out[:4] == 7.0).all()) and bool((out[4 + 3 * int(mol_ptr[-1]):] == 7.0).all())
    for m in good:
        at = slice(3 * int(mol_ptr[m]), 3 * int(mol_ptr[m + 1]))
        assert torch.equal(out[4:-5][at], want[at])
    assert q.device_status() == 0
