"""hc_probe_labels of more queries than it labels at once (131,072), and of slices cut
smaller because the device has no memory for larger ones: the labels of every query are
those of the query asked for alone."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def make(nq):
    from paper_1209_0410_gb300 import datagen, hc
    db = datagen.make_db(30_000, 64, seed=11)
    rows = torch.from_numpy(db).cuda()
    g = torch.Generator(device="cuda").manual_seed(12)
    q = rows[torch.randint(0, 30_000, (nq,), generator=g, device="cuda")].float()
    q = (q + 8 * torch.randn(q.shape, generator=g, device="cuda")).round_().clamp_(0, 255)
    return hc, hc.hc_build(rows, 4, 16), q.to(torch.uint8)


def check(hc, idx, q, labels, k, p_max, at):
    for a in at:
        b = min(a + 500, q.shape[0])
        assert torch.equal(labels[a:b], hc.hc_probe_labels(idx, q[a:b].contiguous(), k, p_max)), a


@pytest.mark.parametrize("nq", [131_072, 131_073, 262_144 + 77])
def test_more_queries_than_a_slice(nq):
    hc, idx, q = make(nq)
    labels = hc.hc_probe_labels(idx, q, 10, 40)
    check(hc, idx, q, labels, 10, 40, (0, 130_800, 131_072 - 250, nq - 500, nq - 77))


class _Props(ctypes.Structure):   # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int),
                ("location_type", ctypes.c_int), ("location_id", ctypes.c_int),
                ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


def test_slices_cut_to_the_memory_there_is():
    """40,000 queries on 256 lists with 128 neighbours need about 90 MB, a memory pool of
    32 MB holds a quarter of them: four times the launches, the same labels."""
    hc, idx, q = make(40_000)
    idx = hc.hc_build(idx.db, 4, 16, partitions=64)

    def run():
        before = hc.hc_launch_count()
        labels = hc.hc_probe_labels(idx, q, 128, 4)
        torch.cuda.synchronize()
        return labels, hc.hc_launch_count() - before

    want, launches = run()
    cuda = ctypes.CDLL("libcuda.so.1")
    default, small = ctypes.c_void_p(), ctypes.c_void_p()
    props = _Props(1, 0, 1, 0, None, 32 << 20, 0)
    assert cuda.cuDeviceGetMemPool(ctypes.byref(default), 0) == 0
    if cuda.cuMemPoolCreate(ctypes.byref(small), ctypes.byref(props)) != 0:
        pytest.skip("no memory pools of a given size here")
    try:
        assert cuda.cuDeviceSetMemPool(0, small) == 0
        labels, more = run()
    finally:
        assert cuda.cuDeviceSetMemPool(0, default) == 0
        assert cuda.cuMemPoolDestroy(small) == 0
    assert more >= 3 * launches and torch.equal(labels, want)
    check(hc, idx, q, labels, 128, 4, (0, 9_700, 39_500))
