"""Events of long units of which little is kept: the selection lists the slots, the assignment the rows that join, and the score pass
writes the defaults.  Against the staged calls, which do none of it: everything must come out the same, byte for byte."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefix,decode,budget,reserve,dup,tau,page", [
    (0, 1601, 100, 100, 0, 0.9, 0),          # no prefix, just sixteen rows a slot
    (900, 3000, 200, 100, 0, 0.9, 16),       # prefix eviction beside it
    (7001, 1030, 500, 60, 0, 0.9, 0),        # little but prefix
    (64, 5000, 200, 136, 3, 0.9, 0),         # three distinct decode keys: ties at the boundaries
    (100, 9000, 300, 250, 1, 0.9, 0),        # more equal scores than a list holds among the decode rows (no lists)
    (6000, 3000, 500, 250, 1, 0.9, 0),       # and in the prefix
    (6000, 3000, 500, 250, 2, 0.9, 0),       # in the prefix alone: seeds out of the row bits
    (700, 9000, 500, 0, 0, 0.9, 0),          # nothing kept of the decode rows but what has to be
    (300, 4000, 200, 150, 0, -1.0, 64),      # every scratch row joins: more members than the list in shared memory holds
    (20, 61420, 900, 700, 0, 0.9, 0),        # the longest unit with lists, two words a thread
    (20, 61421, 900, 700, 0, 0.9, 0),        # and one row more
])
def test_event_equals_the_staged_calls(prefix, decode, budget, reserve, dup, tau, page):
    import gpu_harness as gh
    import torch
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=3, group=2, window=32, prefix=prefix, decode=decode, budget=budget,
                                                reserve=reserve)
    hb = wl.make_batch(w)
    if dup:
        for u in range(hb.n_units):
            a = int(hb.tok_off[u])
            if prefix > 2000:
                hb.k[a:a + prefix] = hb.k[a]
            if dup != 2:
                hb.k[a + prefix:a + prefix + decode] = hb.k[a + prefix + np.arange(decode) % dup]
    run = gh.GpuRun(hb, tau=tau, page_size=page)
    g = run.event()
    assert run.ctx.device_flags() == 0 and run.ctx.used_tensor_path
    st = gh.GpuRun(hb, tau=tau, page_size=page)
    cb, o = st.cb, st.out
    args = (st.ctx, st.batch, st.prm)
    cb.cask_score(*args, o["s"], o["lse"], st.ws, st.ws_bytes)
    cb.cask_prefix_evict(*args, o["s"], o["kind"], o["plan"], st.ws, st.ws_bytes)
    cb.cask_select_core(*args, o["s"], o["plan"], o["kind"], st.ws, st.ws_bytes)
    cb.cask_consolidate_scratch(*args, o["s"], o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"],
                                o["lost_mass"], st.ws, st.ws_bytes)
    cb.cask_compact(*args, o["s"], o["kind"], o["seed_of"], o["weight"], st.out_struct, st.ws, st.ws_bytes)
    torch.cuda.synchronize()
    s = st.numpy_outputs()
    for name in g:
        if name in ("k_out", "v_out"):
            for u in range(hb.n_units):
                k = int(g["n_out"][u])
                assert np.array_equal(g[name][u][:k], s[name][u][:k]), name
        else:
            assert np.array_equal(g[name], s[name]), name
    assert (g["n_out"] == np.minimum(budget, g["plan"][:, 7])).all()


def test_every_unit_of_several_waves_comes_out_the_same():
    """460 copies of one unit, more than the compaction has CTAs on the device at once, with some 1,000 members on 2,000 slots: the later
    CTAs wait for no kernel before them, and their slot counts have to start from zero all the same."""
    import gpu_harness as gh
    copies, T, P, B = 460, 32100, 60, 2000
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=1, group=2, window=32, head_dim=8, prefix=P, decode=T - P, budget=B,
                                                reserve=1990, cluster_frac=0.0)
    k, v, q = wl.make_unit(w, 0, 0, 0)
    hb = wl.Batch(wl=w, k=np.tile(k, (copies, 1)), v=np.tile(v, (copies, 1)), q=np.tile(q[None], (copies, 1, 1, 1)),
                  T=np.full(copies, T, np.int32), P=np.full(copies, P, np.int32), B=np.full(copies, B, np.int32),
                  reserve=np.full(copies, 1990, np.int32), tok_off=np.arange(copies + 1, dtype=np.int64) * T,
                  unit_ids=[(i, 0, 0) for i in range(copies)])
    run = gh.GpuRun(hb, tau=0.9999)
    for _ in range(3):
        g = run.event()
        assert run.ctx.device_flags() == 0
        members = np.isin(g["kind"].reshape(copies, T), (4, 5)).sum(1)
        # (a unit's scores depend in their last bits on the CTAs that share it, so units may differ by a tied row)
        assert (g["n_out"] == B).all() and (members > 950).all() and (members <= 1024).all()
        for u in range(copies):
            a = g["assign"][u * T:(u + 1) * T]
            wt = g["weight"][u * T:(u + 1) * T]
            slots = np.bincount(a[a >= 0], weights=wt[a >= 0], minlength=B)
            assert np.abs(slots - 1.0).max() <= 1e-5, u                      # every slot's weights add up to one
            rows = g["slot_src"][u]
            assert (np.diff(rows) > 0).all() and np.array_equal(a[rows], np.arange(B)), u
            lone = np.bincount(a[a >= 0], minlength=B) == 1
            got = g["k_out"][u][lone]
            assert np.array_equal(got, wl.as_float32(k, w.dtype)[rows[lone]]), u
