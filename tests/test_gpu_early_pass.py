"""The score pass fetches descriptors, keys and queries while the normaliser pass still runs: events of different batches that follow one
another on one workspace, with nothing waited for in between, give the bytes they give alone."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

BF16, FP32 = wl.DTYPE_BF16, wl.DTYPE_FP32
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,window,head_dim,dtype,page,shapes", [
    (4, 128, 128, BF16, 0, [(2, 100, 500), (3, 40, 900), (1, 300, 333)]),         # a few CTAs each, on other SMs every time
    (4, 128, 128, BF16, 16, [(200, 64, 300), (5, 64, 2000), (40, 64, 777)]),      # tables by their own kernel, and by the pass
    (7, 64, 64, BF16, 0, [(9, 100, 3000), (2, 30, 5001)]),                        # two row groups
    (2, 64, 96, FP32, 0, [(2, 100, 900), (7, 64, 1500)]),
])
def test_events_back_to_back_on_one_workspace(group, window, head_dim, dtype, page, shapes):
    import gpu_harness as gh
    import torch
    runs = []
    for units, prefix, decode in shapes:
        w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=group, window=window, prefix=prefix, decode=decode,
                                                    budget=256, reserve=160, dtype=dtype, head_dim=head_dim)
        runs.append(gh.GpuRun(wl.make_batch(w), page_size=page))
    alone = [r.event() for r in runs]
    ws = max((r.ws for r in runs), key=lambda t: t.numel())
    for name in ("s", "kind", "assign", "k_out"):
        for r in runs:
            r.out[name].zero_()
    torch.cuda.synchronize()
    for _ in range(5):
        for r in runs:
            r.cb.cask_compress_event(runs[0].ctx, r.batch, r.prm, r.out_struct, ws, max(x.ws_bytes for x in runs))
    torch.cuda.synchronize()
    for r, want in zip(runs, alone):
        got = r.numpy_outputs()
        for name in ("s", "lse", "kind", "assign", "weight", "slot_src", "k_out", "v_out"):
            assert np.array_equal(got[name], want[name]), name


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
