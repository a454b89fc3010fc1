"""The adjoint of batches that mix many small molecules with a few of 64 atoms or more: the large
ones' centres get a CTA each beside a warp-per-centre launch for the others, with the bits that each
molecule has alone, and a model made for large molecules takes small ones at their own pace."""
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


def _grid_molecule(rng, n):
    """n atoms near the points of a 1.5 A cubic grid."""
    k = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n] * 1.5
    return g + rng.uniform(-0.2, 0.2, size=g.shape), rng.choice(5, size=n).astype(np.int32)


# where the large molecules stand among single atoms: a look covers 2048 molecules in rounds of 256
@pytest.mark.parametrize("n_mol,large", [(1300, {0: 64}), (2100, {255: 65, 256: 200, 2047: 63}),
                                         (2100, {2047: 90, 2048: 64, 2099: 200}),
                                         (4300, {k: 64 + k % 40 for k in range(100, 110)} | {4299: 64})])
def test_large_molecules_among_single_atoms(q, n_mol, large):
    rng = np.random.default_rng(n_mol)
    p = from_table("EF", n2=24, n3=22)
    mols = [_grid_molecule(rng, large.get(k, 1)) for k in range(n_mol)]
    ptr = np.concatenate([[0], np.cumsum([len(e) for _, e in mols])]).astype(np.int32)
    coords = np.concatenate([x for x, _ in mols]).astype(np.float32)
    elem = np.concatenate([e for _, e in mols])
    g = torch.as_tensor(rng.normal(size=(len(elem), q.rep_ld_of(p.rep_dim))).astype(np.float32)).cuda()
    got = q.fchl19_vjp_atoms(coords, elem, ptr, 200, p, g)
    for k, n in large.items():
        at = slice(int(ptr[k]), int(ptr[k + 1]))   # alone: a CTA per centre for every centre
        want = q.fchl19_vjp_atoms(coords[at], elem[at], np.array([0, n], np.int32), 200, p, g[at].contiguous())
        assert torch.equal(got[at], want)
    alone = np.ones(len(elem), bool)
    for k in large:
        alone[ptr[k]:ptr[k + 1]] = False
    assert not got[torch.as_tensor(alone).cuda()].any()   # a single atom feels nothing
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


def test_buffers_for_large_molecules_cost_the_others_little(q):
    """300 molecules of 45 atoms with room for 200: both calls run the same warps on the same centres; the
    rest (a look at 300 sizes, a launch, the reduction's lanes) is a few per cent of ~0.5 ms. A quarter is allowed."""
    rng = np.random.default_rng(1)
    p = from_table("EF", n2=24, n3=22)
    mols = [_grid_molecule(rng, 45) for _ in range(300)]
    ptr = (45 * np.arange(301)).astype(np.int32)
    coords = torch.as_tensor(np.concatenate([x for x, _ in mols]).astype(np.float32)).cuda()
    elem = torch.as_tensor(np.concatenate([e for _, e in mols])).cuda()
    ptr = torch.as_tensor(ptr).cuda()
    g = torch.ones((len(elem), q.rep_ld_of(p.rep_dim)), device="cuda")
    t = [_microseconds(lambda: q.fchl19_vjp_atoms(coords, elem, ptr, mx, p, g)) for mx in (63, 200)]
    assert t[1] <= 1.25 * t[0], t


@pytest.mark.parametrize("n_small", [1000, 20000])
def test_large_molecules_among_pairs(q, n_small):
    """The reduction with eight lanes per output and with one: warps with outputs of small, of large
    and of both kinds of molecules; each large molecule keeps the bits that it has alone."""
    rng = np.random.default_rng(n_small)
    p = from_table("EF", n2=24, n3=22)
    sizes = np.full(n_small, 2)
    sizes[[0, 7, 8, 500, n_small - 2]] = 66, 64, 200, 63, 91
    mols = [_grid_molecule(rng, n) for n in sizes]
    ptr = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    coords = np.concatenate([x for x, _ in mols]).astype(np.float32)
    elem = np.concatenate([e for _, e in mols])
    g = torch.as_tensor(rng.normal(size=(len(elem), q.rep_ld_of(p.rep_dim))).astype(np.float32)).cuda()
    got = q.fchl19_vjp_atoms(coords, elem, ptr, 200, p, g)
    for k in [0, 1, 6, 7, 8, 9, 500, n_small - 2, n_small - 1]:
        at = slice(int(ptr[k]), int(ptr[k + 1]))
        want = q.fchl19_vjp_atoms(coords[at], elem[at], np.array([0, sizes[k]], np.int32), 200, p, g[at].contiguous())
        assert torch.equal(got[at], want)
    assert q.device_status() == 0


def test_reduction_of_small_molecules_with_room_for_large_ones(q):
    """12 000 molecules of 18 atoms with room for 200 against room for 29: the same centres and sums, beside a look
    at 12 000 sizes and a launch, ~10 us of ~1 ms. A quarter is allowed."""
    rng = np.random.default_rng(2)
    p = from_table("EF", n2=24, n3=22)
    mols = [_grid_molecule(rng, 18) for _ in range(12000)]
    ptr = torch.as_tensor((18 * np.arange(12001)).astype(np.int32)).cuda()
    coords = torch.as_tensor(np.concatenate([x for x, _ in mols]).astype(np.float32)).cuda()
    elem = torch.as_tensor(np.concatenate([e for _, e in mols])).cuda()
    g = torch.ones((len(elem), q.rep_ld_of(p.rep_dim)), device="cuda")
    t = [_microseconds(lambda: q.fchl19_vjp_atoms(coords, elem, ptr, mx, p, g)) for mx in (29, 200)]
    assert t[1] <= 1.25 * t[0], t
