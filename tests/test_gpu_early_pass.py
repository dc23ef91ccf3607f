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
