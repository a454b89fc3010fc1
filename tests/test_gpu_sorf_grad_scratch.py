"""qmlr_sorf_grad takes no memory under stream capture and has the same bits with and without its scratch."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2206_01580_gb300 import synth

pytestmark = pytest.mark.gpu

MEM_ALLOC, MEM_FREE = 10, 11   # cudaGraphNodeTypeMemAlloc, cudaGraphNodeTypeMemFree


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_01580_gb300 import qmlr
    qmlr.lib()
    return qmlr


@pytest.mark.parametrize("d,n_features,n_atoms", [(16, 48, 129), (64, 512, 300), (128, 128 * 130, 140)])
@pytest.mark.parametrize("forces", [True, False])
def test_captured_call_owns_no_memory(q, d, n_features, n_atoms, forces):
    rng = np.random.default_rng(n_features)
    signs, b = synth.sorf_draw(rng, n_features, d, 3)
    sb = q.pack_signs(signs)
    b = torch.as_tensor(b.astype(np.float32)).cuda()
    alpha = torch.as_tensor(rng.normal(size=n_features).astype(np.float32)).cuda()
    x = torch.as_tensor(rng.normal(size=(n_atoms, d)).astype(np.float32)).cuda()
    ptr = torch.tensor([0, 40, n_atoms], dtype=torch.int32, device="cuda")
    want_e, want_g = q.sorf_grad(x, ptr, sb, 3, b, 2.0, alpha)   # more than 128 atoms: with scratch
    parts = q.sorf_parts(n_features, d)
    e_atom = torch.zeros((parts, n_atoms), device="cuda", dtype=torch.float64)
    e = torch.zeros(2, device="cuda", dtype=torch.float64)
    g = torch.zeros((parts, n_atoms, d), device="cuda")
    rt = C.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        s = C.c_void_p(stream.cuda_stream)
        assert rt.cudaStreamBeginCapture(s, C.c_int(2)) == 0   # cudaStreamCaptureModeRelaxed
        rc = q.lib().qmlr_sorf_grad(q._ptr(x), d, q._ptr(ptr), 2, n_atoms, q._ptr(sb), 3, q._ptr(b), n_features, 2.0,
                                    q._ptr(alpha), q._ptr(e_atom), q._ptr(e), q._ptr(g) if forces else None, s)
        graph = C.c_void_p()
        assert rt.cudaStreamEndCapture(s, C.byref(graph)) == 0 and rc == 0
    n = C.c_size_t(0)
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0 and n.value > 0
    nodes = (C.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
    for node in nodes:
        kind = C.c_int(-1)
        assert rt.cudaGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        assert kind.value not in (MEM_ALLOC, MEM_FREE)
    run = C.c_void_p()
    assert rt.cudaGraphInstantiate(C.byref(run), graph, C.c_ulonglong(0)) == 0
    assert rt.cudaGraphLaunch(run, s) == 0
    stream.synchronize()
    assert torch.equal(e, want_e)
    if forces:
        assert torch.equal(g, want_g)
    assert rt.cudaGraphExecDestroy(run) == 0 and rt.cudaGraphDestroy(graph) == 0
    assert q.device_status() == 0


@pytest.mark.parametrize("n_atoms", [1, 128, 129])
def test_same_bits_on_both_sides_of_the_rule(q, n_atoms):
    """Atoms are independent: a batch on either side of the 128-atom rule has the bits of a larger batch's first atoms."""
    rng = np.random.default_rng(3)
    signs, b = synth.sorf_draw(rng, 1024, 128, 3)
    sb, al = q.pack_signs(signs), rng.normal(size=1024).astype(np.float32)
    x = torch.as_tensor(rng.normal(size=(200, 128)).astype(np.float32)).cuda()
    ptr = lambda n: torch.arange(n + 1, dtype=torch.int32, device="cuda")
    e, g = q.sorf_grad(x, ptr(200), sb, 3, b.astype(np.float32), 2.0, al)
    e1, g1 = q.sorf_grad(x[:n_atoms].contiguous(), ptr(n_atoms), sb, 3, b.astype(np.float32), 2.0, al)
    assert torch.equal(e1, e[:n_atoms]) and torch.equal(g1, g[:, :n_atoms])
    assert q.device_status() == 0
