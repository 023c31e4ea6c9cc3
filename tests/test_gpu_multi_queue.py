"""The multi-set tensor counts' queue: units decoded a warp at a time, the set
found by a 32-way search.  Histograms are integers: equal to the POPC path's."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [2, 3])
@pytest.mark.parametrize("sizes", [[1], [2], [257] * 3, [1, 2, 255, 256, 257, 512, 513], list(range(1, 34)),
                                   [3 + (7 * s) % 300 for s in range(1100)], [2300, 1, 4000, 2, 1800]])
def test_sets_of_every_span(path, sizes):
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    sets = [((2, 4, 3)[s % 3], n, 100 + s) for s, n in enumerate(sizes)]
    hists = []
    for p in (1, path):
        b = cs.Batch(sets, path=p, n_eps=0)
        b.launch(())
        assert b.status() == 0
        hists.append(b.hist.cpu())
    assert torch.equal(*hists)


@pytest.mark.parametrize("path", [2, 3])
def test_slices_with_empty_ones_between(path):
    """Count jobs over slices of several sets, empty slices first, last and in a row."""
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    bufs, ops = [], []
    for s, n in enumerate((300, 1500, 700, 2600)):
        b = cs.allocate(2, n, path=1)
        cs.run(b, 40 + s, eps=())
        nb = cs.operands_bytes(n, path)
        o = torch.empty(nb + 1024, dtype=torch.uint8, device="cuda")
        ptr = (o.data_ptr() + 1023) // 1024 * 1024
        cs.prepare_operands(n, b.bits, ptr, nb, path=path)
        bufs.append((b, o, ptr, torch.zeros_like(b.hist)))
    jobs, L = [], cs.lib()
    for step in range(7):
        for b, o, ptr, h in bufs:
            total = cs.count_items(b.n, path)
            lo, hi = total * step // 7, total * (step + 1) // 7
            if path == 2:  # whole supertiles only matter for the pair path; any slice is fine here
                lo, hi = min(lo, total), min(hi, total)
            jobs += [cs.CountJob(b.bits.data_ptr(), b.n, b.rw, h.data_ptr(), ptr, x, y)
                     for x, y in ((lo, lo), (lo, hi), (hi, hi))]
    tab = torch.empty(L.cs_count_jobs_table_bytes(len(jobs), path) + 128, dtype=torch.uint8, pin_memory=True)
    ws = torch.empty(L.cs_count_jobs_workspace_bytes(len(jobs), path), dtype=torch.uint8, device="cuda")
    cs.count_jobs(jobs, path, (tab.data_ptr() + 127) // 128 * 128, ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    for b, o, ptr, h in bufs:
        assert torch.equal(h, b.hist), b.n
