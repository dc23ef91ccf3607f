"""The scoring passes read a block table for several tiles at once, a batch ahead: scores and normalisers of a paged cache are those of the
same rows one behind the other, bit for bit."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("page,group,window,units,T", [
    (8, 1, 64, 3, 2000),            # two tiles a batch
    (16, 4, 64, 200, 517),          # four; units of five tiles, shared by CTAs anywhere
    (32, 7, 64, 5, 3001),
    (64, 1, 64, 160, 2500),         # sixteen: a segment and a rest of four
    (128, 2, 64, 150, 4300),        # thirty-two, of a segment of thirty-four
    (256, 4, 128, 150, 4300),       # a page is two tiles
    (16, 8, 128, 40, 1100),         # two row groups: a unit's pages twice
])
def test_scores_of_paged_rows(page, group, window, units, T):
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=1, group=group, window=window, prefix=100, decode=T - 100, budget=256, reserve=160)
    k, v, q = wl.make_unit(w, 0, 0, 0)
    rng = np.random.default_rng(page)
    lens = (T - rng.integers(0, T // 3, units) * (units > 10)).astype(np.int32)         # ragged where there are many
    tok = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    full = lambda x: np.full(units, x, np.int32)
    cut = lambda a: np.concatenate([np.roll(a, 37 * u, 0)[:t] for u, t in enumerate(lens)])
    hb = wl.Batch(wl=w, k=cut(k), v=cut(v), q=np.tile(q[None], (units, 1, 1, 1)), T=lens, P=full(100), B=full(256), reserve=full(160), tok_off=tok,
                  unit_ids=[(i, 0, 0) for i in range(units)])
    outs = []
    for ps in (0, page):
        run = gh.GpuRun(hb, page_size=ps)
        run.cb.cask_score(run.ctx, run.batch, run.prm, run.out["s"], run.out["lse"], run.ws, run.ws_bytes)
        assert run.ctx.device_flags() == 0 and run.ctx.used_tensor_path
        outs.append((run.out["s"].cpu().numpy(), run.out["lse"].cpu().numpy()))
    assert all(np.array_equal(a.view(np.uint8), b.view(np.uint8)) for a, b in zip(*outs))
    assert np.isfinite(outs[0][0]).all() and abs(float(outs[0][0].sum()) - units) < 1e-3 * units
