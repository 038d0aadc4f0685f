"""Batches in arrival order whose last wave is nearly full, on rows at the reach of an
SM's address translation, ask for ids behind rows: their results at and beside the lines
of that rule equal those of small batches."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mb,d,parts,k,p", [(245, 128, 1, 10, 40), (245, 64, 1, 32, 33),
                                            (500, 128, 2, 1, 17), (330, 128, 1, 10, 1),
                                            (330, 64, 1, 7, 300)])
def test_full_waves_equal_small_batches(mb, d, parts, k, p):
    from paper_1209_0410_gb300 import hc
    wave = 24 * torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(mb + d)
    n = (mb << 20) // d + 3
    db = torch.randint(0, 256, (n, d), generator=g, device="cuda", dtype=torch.uint8)
    q = db[torch.randint(0, n, (5 * wave + 1,), generator=g, device="cuda")].contiguous()
    q[::9] = 255
    idx = hc.hc_build(db, d // 16, 16, partitions=parts)
    small = [hc.hc_query(idx, q[a:a + 2000].contiguous(), k, p) for a in range(0, len(q), 2000)]
    want = [torch.cat([s[i] for s in small]) for i in (0, 1)]
    for nq in (wave * 66 // 100, wave * 66 // 100 + 1, wave, wave + 1, wave * 9 // 5, 2 * wave,
               3 * wave, 3 * wave + 1, 5 * wave, 5 * wave + 1):
        got = hc.hc_query(idx, q[:nq].contiguous(), k, p)
        assert all(torch.equal(got[i], want[i][:nq]) for i in (0, 1)), nq
