"""To 128 seeds and from tau = 0.5 up, the tensor-core assignment looks for a row's greatest cosine first, sixteen seeds at a time, and for the seed
it belongs to only where the row joins.  Caches of few distinct keys, each many times among the seeds: the first seed among equals wins, in
whichever sixteen it lies.  The SIMT kernel is the reference."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl
from test_gpu_many_seeds import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [0.9, 0.5, 0.49])                       # the last by the search in every sixteen
@pytest.mark.parametrize("m,head_dim,page,units", [
    (1, 128, 0, 3), (15, 128, 16, 3), (16, 64, 0, 3), (17, 128, 0, 200),
    (95, 128, 0, 3), (96, 128, 64, 3), (97, 80, 0, 3), (112, 64, 16, 40), (127, 128, 0, 3), (128, 128, 0, 3), (129, 128, 0, 3), (256, 64, 0, 3),
])
def test_first_seed_among_equals(m, head_dim, page, units, tau):
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=4, window=32, prefix=50, decode=1200, budget=50 + 32 + 2 * m,
                                                reserve=32 + 2 * m, head_dim=head_dim)
    hb = wl.make_batch(w)
    rng = np.random.default_rng(m)
    k = hb.k.reshape(units, 1250, -1)
    for u in range(units):
        k[u, 50:1000] = k[u, 50 + rng.integers(0, min(40, m), 950)]     # some forty distinct keys, then rows of their own
    a = _compare(hb, page, tau=tau)
    assert (a["plan"][:, 5] == m).all()
    assert m < 15 or ((a["kind"] == 5).any() and (a["kind"] == 0).any())


@pytest.mark.parametrize("m", [96, 200])
def test_the_reference_is_another_kernel(m):
    """The two sum 128 products in another order, so that some cosine differs: what is compared above is not one kernel with itself."""
    import gpu_harness as gh
    hb = wl.make_batch(wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=3, group=4, window=32, prefix=50, decode=1200, budget=82 + 2 * m, reserve=32 + 2 * m))
    run = gh.GpuRun(hb)
    o, args, ws, sims = run.out, (run.ctx, run.batch), (run.ws, run.ws_bytes), []
    run.cb.cask_score(*args, run.prm, o["s"], o["lse"], *ws)
    for prm in (run.prm, run.cb.params(score_path=1)):
        run.cb.cask_prefix_evict(*args, run.prm, o["s"], o["kind"], o["plan"], *ws)
        run.cb.cask_select_core(*args, run.prm, o["s"], o["plan"], o["kind"], *ws)
        run.cb.cask_consolidate_scratch(*args, prm, o["s"], o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"], o["lost_mass"], *ws)
        sims.append(o["sim"].cpu().numpy())
    assert (o["plan"][:, 5] == m).all() and (sims[0] != sims[1]).any() and np.abs(sims[0] - sims[1]).max() <= 2 * 128 * 2.0 ** -24
