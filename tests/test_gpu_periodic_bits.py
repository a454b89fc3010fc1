"""Periodic FCHL19 by a CTA per centre and by a warp per centre on one system: the forward has the same bits."""
import copy

import numpy as np
import pytest
import torch

from paper_2206_01580_gb300 import synth
from paper_2206_01580_gb300.params import from_table

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr
    qmlr.lib()
    return qmlr


def _copies(s, k):
    """k copies of a system that do not see each other: the same positions and shifts, environments of their own."""
    t = copy.copy(s)
    n, e = s.n_atoms, s.n_entries
    t.n_atoms, t.n_entries = k * n, k * e
    t.coords, t.elem = s.coords.repeat(k, 1), s.elem.repeat(k)
    at = torch.arange(k, device="cuda").repeat_interleave(e)
    t.env_atom = (s.env_atom.repeat(k) + at * n).to(torch.int32)
    t.env_shift = s.env_shift.repeat(k, 1)
    t.env_ptr = torch.cat([s.env_ptr[:1]] + [s.env_ptr[1:] + j * e for j in range(k)])
    return t


def test_many_centres_have_the_bits_of_few(q):
    """12 800 centres (beyond 12 288 a warp each) against 1600 (a CTA each), ~70 entries per centre."""
    p = from_table("EF", n2=24, n3=22)
    s = synth.framework_crystal(np.random.default_rng(3), 1600)
    system = q.PeriodicSystem(s.coords, s.elem, s.cell, p.rcut)
    assert system.max_env >= 32
    few, many = q.fchl19_periodic(system, p), q.fchl19_periodic(_copies(system, 8), p)
    assert q.device_status() == 0
    assert torch.equal(many, few.repeat(8, 1))


def test_room_for_many_entries_has_the_bits_of_few(q):
    """Fewer than 32 entries per centre (a warp each), and the same with room for 64 (a CTA each)."""
    p = from_table("EF", n2=24, n3=22)
    s = synth.framework_crystal(np.random.default_rng(5), 60, density=0.015)
    system = q.PeriodicSystem(s.coords.astype(np.float32), s.elem, s.cell, p.rcut)
    assert 0 < system.max_env < 32
    few = q.fchl19_periodic(system, p)
    system.max_env = 64
    assert torch.equal(q.fchl19_periodic(system, p), few)
    assert q.device_status() == 0


def _microseconds(f):
    for _ in range(3):
        f()
    best = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b) * 200.0)
    return min(best)


def test_room_for_dense_places_costs_a_sparse_system_little(q):
    """12 000 centres with fewer than 32 entries, and the same with room for 64: the mean stays what it is, and the
    kernels for dense systems return at once, a launch and 12 000 CTAs (~5 us) beside ~60. A third is allowed."""
    p = from_table("EF", n2=24, n3=22)
    s = synth.framework_crystal(np.random.default_rng(5), 60, density=0.015)
    few = _copies(q.PeriodicSystem(s.coords.astype(np.float32), s.elem, s.cell, p.rcut), 200)
    room = copy.copy(few)
    room.max_env = 64
    assert 0 < few.max_env < 32
    t = [_microseconds(lambda: q.fchl19_periodic(x, p)) for x in (few, room)]
    assert t[1] <= 4.0 / 3.0 * t[0], t
