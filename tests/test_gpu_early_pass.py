"""The score pass fetches descriptors, block table, keys and queries while the normaliser pass still runs: events of different batches that
follow one another on one workspace, each behind kernels that rewrite its cache, queries and block table in place, give what they
give alone, and the scores of the SIMT kernels."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

BF16, FP32 = wl.DTYPE_BF16, wl.DTYPE_FP32
pytestmark = pytest.mark.gpu


def _contents(run):
    """Two contents of a run's cache, queries and block table, of the same sizes.  A paged cache has its pages in other places in the second
    one, so that a table of the one with a pool of the other is another cache; a contiguous one its rows in reverse order."""
    torch, dev = run.torch, run.dev
    first = [(dev[n], dev[n].clone()) for n in ("k", "v", "q")]
    second = [(dev["q"], dev["q"].flip(0).contiguous())]
    if run.batch.page_size:
        ps = run.batch.page_size
        n = dev["k"].shape[0] // ps
        to = torch.from_numpy(np.random.default_rng(5).permutation(n)).to(dev["k"].device)          # page p moves to to[p]
        for name in ("k", "v"):
            moved = torch.empty_like(dev[name])
            moved.view(n, ps, -1)[to] = dev[name].view(n, ps, -1)
            second.append((dev[name], moved))
        first.append((run.block_table, run.block_table.clone()))
        second.append((run.block_table, to[run.block_table.long()].to(torch.int32)))
    else:
        second += [(dev[name], dev[name].flip(0).contiguous()) for name in ("k", "v")]
    return first, second


@pytest.mark.parametrize("group,window,head_dim,dtype,page,shapes", [
    (4, 128, 128, BF16, 0, [(2, 100, 500), (3, 40, 900), (1, 300, 333)]),         # a few CTAs each, on other SMs every time
    (4, 128, 128, BF16, 16, [(200, 64, 300), (5, 64, 2000), (40, 64, 777)]),      # tables by their own kernel, and by the pass
    (7, 64, 64, BF16, 0, [(9, 100, 3000), (2, 30, 5001)]),                        # 448 rows: three and a half blocks
    (4, 64, 128, BF16, 64, [(9, 100, 3000), (150, 30, 700)]),                     # two blocks a tile
    (1, 100, 80, BF16, 0, [(9, 100, 3000), (2, 30, 5001)]),                       # one block
    (7, 128, 128, BF16, 0, [(9, 100, 3000), (80, 30, 700)]),                      # 896 rows: two row groups, their tables by both ways
    (12, 65, 80, BF16, 128, [(3, 100, 3000), (100, 30, 700)]),                    # 780 rows: two row groups
    (2, 64, 96, FP32, 0, [(2, 100, 900), (7, 64, 1500)]),
    (4, 64, 128, FP32, 0, [(3, 100, 900), (80, 64, 500)]),                        # two row groups of fp32
])
def test_events_back_to_back_on_one_workspace(group, window, head_dim, dtype, page, shapes):
    import gpu_harness as gh
    import torch
    runs = []
    for units, prefix, decode in shapes:
        w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=group, window=window, prefix=prefix, decode=decode,
                                                    budget=256, reserve=160, dtype=dtype, head_dim=head_dim)
        runs.append(gh.GpuRun(wl.make_batch(w), page_size=page))
    ws = max((r.ws for r in runs), key=lambda t: t.numel())
    ws_bytes = max(r.ws_bytes for r in runs)
    bits = lambda t: t.contiguous().view(torch.uint8)

    def event(r, content, prm):
        for dst, src in content:
            dst.copy_(src)
        for t in r.out.values():
            bits(t).fill_(0xA5)
        r.cb.cask_compress_event(runs[0].ctx, r.batch, prm, r.out_struct, ws, ws_bytes)
        return {name: t.clone() for name, t in r.out.items()}

    work = [(r, c) for r in runs for c in _contents(r)]
    want = []
    simt = runs[0].cb.params(score_path=1)
    for r, c in work:
        # alone, with an event recorded between any two kernels: none starts before the one ahead of it has ended
        torch.cuda.synchronize()
        runs[0].ctx.profile_enable(True)
        want.append(event(r, c, r.prm))
        torch.cuda.synchronize()
        runs[0].ctx.profile_enable(False)
        assert runs[0].ctx.device_flags() == 0 and runs[0].ctx.score_path != 0
        s = event(r, c, simt)["s"]
        assert torch.allclose(want[-1]["s"], s, rtol=gh.SCORE_RTOL, atol=1e-12)
    assert not torch.equal(want[0]["s"], want[1]["s"])
    torch.cuda.synchronize()
    got = [[event(r, c, r.prm) for r, c in work] for _ in range(5)]
    torch.cuda.synchronize()
    for n, outs in enumerate(got):
        for g, w in zip(outs, want):
            for name in w:
                assert torch.equal(bits(g[name]), bits(w[name])), (n, name)


def test_descriptors_leave_before_the_normaliser_pass_comes():
    """The descriptor kernel starts beside the compaction of the event before, whose CTAs fill the chip but for a few places at three
    units an SM.  A few units fewer take no longer (3 % longer when the pass that follows started beside the descriptor kernel)."""
    import gpu_harness as gh
    import torch
    places = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    w = wl.WORKLOADS["serving_steady_b512"].with_(layers=1, kv_heads=1, n_seqs=1, group=4, window=128, prefix=200, decode=440, budget=512, reserve=200)
    k, v, q = wl.make_unit(w, 0, 0, 0)
    runs = []
    for n in (places - 12, places):
        full = lambda x: np.full(n, x, np.int32)
        runs.append(gh.GpuRun(wl.Batch(wl=w, k=np.tile(k, (n, 1)), v=np.tile(v, (n, 1)), q=np.tile(q[None], (n, 1, 1, 1)), T=full(640),
                                       P=full(200), B=full(512), reserve=full(200), tok_off=np.arange(n + 1, dtype=np.int64) * 640,
                                       unit_ids=[(i, 0, 0) for i in range(n)])))
        runs[-1].out_struct.rho_core = runs[-1].out_struct.rho_rep = runs[-1].out_struct.dispersion = None        # (no diagnostics)
    times = [[], []]
    for _ in range(9):
        for r, t in zip(runs, times):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for i in range(43):
                if i == 3:
                    a.record()
                r.cb.cask_compress_event(r.ctx, r.batch, r.prm, r.out_struct, r.ws, r.ws_bytes)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
    assert np.median(times[0]) < 1.01 * np.median(times[1]), times
