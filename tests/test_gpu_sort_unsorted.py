"""The allocation-free sort on stores in random order, in calls that follow one another without a synchronisation:
the calls share their scratch, so the offsets that one reads lie where another's lay before (rows of cells that do
not fill a cache line, too). Bit for bit against a stable sort."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [3, 101, 512, 2047, 4096])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_consecutive_sorts_of_random_stores(prec, cells):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import _native as NV, pic
    real = torch.float32 if prec == "fp32" else torch.float64
    code = pic.FP32 if prec == "fp32" else pic.FP64
    gen = torch.Generator(device="cuda").manual_seed(cells)
    calls = []
    for n in (300_001, 4096, 300_001, 77_777, 500_000, 31):
        c = torch.randint(0, cells, (n,), generator=gen, device="cuda").to(torch.int32)
        if n % 2 == 0:  # few of the cells, in descending order
            c = torch.sort(c // 2, descending=True).values.contiguous()
        r = torch.randn((n, 4), generator=gen, device="cuda", dtype=real)
        calls.append((c, r, torch.empty_like(c), torch.empty_like(r)))
    torch.cuda.synchronize()
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for c, r, co, ro in calls * 2:
        NV.check(NV.lib().pic_sort_noalloc(*[C.c_void_p(t.data_ptr()) for t in (c, r, co, ro)], c.numel(), cells, code, st))
    torch.cuda.synchronize()
    for c, r, co, ro in calls:
        want, at = torch.sort(c, stable=True)
        assert torch.equal(co, want) and torch.equal(ro, r[at]), c.numel()
