"""Chain tables given with a FeatureSpec: the same features and rows as with the tables of the call."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2206_01580_gb300 import pipeline, qmlr, synth
from paper_2206_01580_gb300.params import from_table

pytestmark = pytest.mark.gpu


def test_given_tables():
    rng = np.random.default_rng(8)
    p = from_table("EF", n2=24, n3=22)
    mols = synth.random_box(rng, 5, 9)
    signs, b = synth.sorf_draw(rng, 512, 128, 2)
    spec = pipeline.spec_from(p, 128, signs, b.astype(np.float32), 2.0)
    U = torch.as_tensor(rng.normal(size=(5, p.rep_dim, 128)).astype(np.float32) * 0.05).cuda()
    batch = pipeline.Batch.from_host(mols.coords, mols.elem, mols.mol_ptr)
    given = dataclasses.replace(spec, tc_tables=qmlr.sorf_tc_tables(spec.sign_bits, 2, 512))
    assert torch.equal(pipeline.feature_matrix(batch, given, U), pipeline.feature_matrix(batch, spec, U))
    assert torch.equal(pipeline.energy_force_rows(batch, given, U), pipeline.energy_force_rows(batch, spec, U))
    assert spec.tc_tables is None
    assert qmlr.device_status() == 0
