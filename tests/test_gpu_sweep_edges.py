"""Sweeps of ascending ids, on batches that take them: the largest number of lists
whose positions fit beside a second block (96, and 104 past it), blocks with few queries,
windows cut off at both ends of every list, lists of up to 64 neighbours.  The walk each
batch takes is read from the names of its kernels.  (The choice of the walk keeps
windows of fewer than 1,024 entries, and with them empty walks, off the sweeps.)"""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def kernels_of(fn, path):
    """The text of the names of the kernels fn(stream) launches (of a captured graph)."""
    cuda, graph, stream = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    torch.cuda.synchronize()
    assert cuda.cuStreamBeginCapture_v2(handle, 1) == 0
    fn(stream)
    assert cuda.cuStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert cuda.cuGraphDebugDotPrint(graph, str(path).encode(), 1) == 0
    assert cuda.cuGraphDestroy(graph) == 0
    return path.read_text()


@pytest.mark.parametrize("mb,d,curves,parts,k,p,over,sweeps", [
    (350, 128, 8, 1, 10, 64, 1, True), (350, 128, 8, 1, 10, 63, 1, False),
    (350, 128, 8, 1, 64, 200, 7, True), (350, 128, 8, 1, 64, 199, 7, False),
    (350, 128, 3, 1, 32, 1000, 5, True), (2430, 128, 8, 12, 10, 6, 3, True),
    (2430, 128, 8, 12, 33, 17, 6, True), (2640, 128, 8, 13, 10, 6, 3, False),
    (530, 48, 3, 1, 1, 200, 2, True)])
def test_sweeps(tmp_path, mb, d, curves, parts, k, p, over, sweeps):
    from paper_1209_0410_gb300 import hc
    nq = 4 * torch.cuda.get_device_properties(0).multi_processor_count * 16 + over
    g = torch.Generator(device="cuda").manual_seed(mb + d + p)
    n = (mb << 20) // d + 5
    db = torch.empty((n, d), dtype=torch.uint8, device="cuda")
    for a in range(0, n, 1 << 21):
        db[a:a + (1 << 21)] = torch.randint(0, 256, db[a:a + (1 << 21)].shape, generator=g,
                                            device="cuda", dtype=torch.uint8)
    q = db[torch.randint(0, n, (nq,), generator=g, device="cuda")].contiguous()
    q[::7] = 0        # the first of every list
    q[3::11] = 255
    idx = hc.hc_build(db, curves, 16, partitions=parts)
    first = hc.hc_query_positions(idx, q[:1].contiguous())
    assert int(first.max()) == 0
    small = [hc.hc_query(idx, q[a:a + 2500].contiguous(), k, p) for a in range(0, nq, 2500)]
    space = torch.empty(hc.hc_query_ordered_workspace(idx, nq), dtype=torch.uint8, device="cuda")
    got = hc.hc_query_ordered(idx, q, k, p, workspace=space)
    names = kernels_of(lambda stream: hc.hc_query_ordered(idx, q, k, p, *got, space, stream),
                       tmp_path / "graph.dot")
    assert ("sweep_kernel" in names) == sweeps and ("query_kernel" in names) != sweeps
    assert all(torch.equal(got[i], torch.cat([s[i] for s in small])) for i in (0, 1))
