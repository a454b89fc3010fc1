"""force_rows_tc refuses outputs of another layout on the host."""
import pytest
import torch

D, NF, T = 128, 256, 3


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
