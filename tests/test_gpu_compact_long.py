"""The one-kernel compaction of longer units at its edges, against the oracle: misaligned row offsets, row counts around its
passes, head dims of every form, thousands of members, budgets of one slot to more than the cache, few units and many."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype,tau,page", [
    (128, wl.DTYPE_BF16, 0.9, 0),
    (64, wl.DTYPE_BF16, -1.0, 0),        # every scratch row merges: thousands of members
    (80, wl.DTYPE_BF16, 0.9, 16),
    (8, wl.DTYPE_BF16, 0.5, 0),
    (128, wl.DTYPE_FP32, -1.0, 0),
    (200, wl.DTYPE_FP32, 0.9, 48),
])
def test_edges(d, dtype, tau, page):
    import gpu_harness as gh
    base = wl.WORKLOADS["tiny"].with_(dtype=dtype, head_dim=d, group=2, window=16, cluster_frac=0.7, n_centres=0)
    # (rows, prefix, budget, reserve): odd lengths, so that the units after the first start at every alignment
    specs = [(4096, 0, 20, 20), (4097, 300, 64, 40), (16, 3, 5, 3), (1025, 1, 1030, 8), (8191, 8000, 700, 30), (4079, 0, 600, 600),
             (33, 33, 9, 2), (2050, 100, 2049, 1949), (1500, 700, 1, 0)]
    parts = [wl.make_unit(base.with_(prefix=p, decode=t - p), i, 0, 0) for i, (t, p, b, r) in enumerate(specs)]
    T, P, B, R = (np.array(x, np.int32) for x in zip(*specs))
    hb = wl.Batch(wl=base, k=np.concatenate([p[0] for p in parts]), v=np.concatenate([p[1] for p in parts]),
                  q=np.stack([p[2] for p in parts]), T=T, P=P, B=B, reserve=R,
                  tok_off=np.concatenate([[0], np.cumsum(T)]).astype(np.int64), unit_ids=[(i, 0, 0) for i in range(len(T))])
    run = gh.GpuRun(hb, tau=tau, page_size=page)
    g = run.event()
    assert run.ctx.device_flags() == 0
    st = gh.compare_event(hb, g, gh.run_oracle(hb, tau=tau), tau=tau)
    assert st["cascaded"] <= 1 and st["merged_elems"] > 0
    for u in range(len(specs)):
        k = int(g["n_out"][u])
        assert (g["slot_src"][u][k:] == -1).all() and (g["slot_kind"][u][k:] == 0).all() and (g["slot_mass"][u][k:] == 0).all()
        assert (np.diff(g["slot_src"][u][:k]) > 0).all()
    again = gh.GpuRun(hb, tau=tau, page_size=page).event()
    for name in g:
        if name not in ("k_out", "v_out"):
            assert np.array_equal(g[name], again[name]), name


@pytest.mark.parametrize("copies", [1, 60, 600])
def test_every_division_of_a_unit_among_ctas_gives_the_same(copies):
    """A unit's slots are shared out among up to sixteen CTAs when there are few units: the same bytes as with one."""
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=1, group=2, window=16, prefix=100, decode=1300, budget=200,
                                                reserve=120)
    k, v, q = wl.make_unit(w, 0, 0, 0)
    T = 1400
    hb = wl.Batch(wl=w, k=np.tile(k, (copies, 1)), v=np.tile(v, (copies, 1)), q=np.tile(q[None], (copies, 1, 1, 1)),
                  T=np.full(copies, T, np.int32), P=np.full(copies, 100, np.int32), B=np.full(copies, 200, np.int32),
                  reserve=np.full(copies, 120, np.int32), tok_off=np.arange(copies + 1, dtype=np.int64) * T,
                  unit_ids=[(i, 0, 0) for i in range(copies)])
    s = np.linspace(0.0, 1.0, T).astype(np.float32)[np.random.default_rng(1).permutation(T)]
    run = gh.GpuRun(hb)
    cb, o = run.cb, run.out
    s_dev = run.dev_f32(np.tile(s, copies))
    args = (run.ctx, run.batch, run.prm)
    cb.cask_prefix_evict(*args, s_dev, o["kind"], o["plan"], run.ws, run.ws_bytes)
    cb.cask_select_core(*args, s_dev, o["plan"], o["kind"], run.ws, run.ws_bytes)
    cb.cask_consolidate_scratch(*args, s_dev, o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"],
                                o["lost_mass"], run.ws, run.ws_bytes)
    cb.cask_compact(*args, s_dev, o["kind"], o["seed_of"], o["weight"], run.out_struct, run.ws, run.ws_bytes)
    run.torch.cuda.synchronize()
    g = run.numpy_outputs()
    for name in ("k_out", "v_out", "slot_src", "slot_kind", "slot_mass", "n_out"):
        for u in range(1, copies):
            assert np.array_equal(g[name][u], g[name][0]), (name, u)
    for name in ("assign", "weight", "kind", "seed_of"):
        x = g[name].reshape(copies, T)
        assert (x == x[0]).all(), name
    kd = g["kind"][:T]
    assert (kd == 5).any() and int(g["n_out"][0]) == int((np.isin(kd, (1, 2, 3, 4))).sum()) == 200
    keep = np.nonzero(np.isin(kd, (1, 2, 3, 4)))[0]
    assert np.array_equal(g["slot_src"][0], keep) and np.array_equal(g["assign"][:T][keep], np.arange(200))
    kf = wl.as_float32(k, w.dtype)
    for t in np.nonzero(kd[keep] == 4)[0]:
        mem = np.nonzero(g["assign"][:T] == t)[0]
        want = (g["weight"][:T][mem, None].astype(np.float64) * kf[mem]).sum(0)
        assert np.abs(g["k_out"][0][t] - want).max() <= np.maximum(2e-2, np.abs(want) * 2.0 ** -7).max()


def test_thousands_of_members_cost_a_fraction_more():
    """An event in which every scratch row joins against one in which none does: more rows to add up, which takes about twice the
    time (it was nine times when every group's warp looked through all of the unit's members)."""
    import gpu_harness as gh
    import torch
    hb = wl.make_batch(wl.WORKLOADS["reasoning8k_b512"].with_(layers=4, kv_heads=4))

    def best_ms(tau):
        run = gh.GpuRun(hb, tau=tau)
        run.out_struct.rho_core = run.out_struct.rho_rep = run.out_struct.dispersion = None        # (no diagnostics)
        run.event()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                run.cb.cask_compress_event(run.ctx, run.batch, run.prm, run.out_struct, run.ws, run.ws_bytes)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        members = np.isin(run.out["kind"].cpu().numpy(), (4, 5)).sum() / hb.n_units
        return min(times), members

    (all_join, many), (none_joins, few) = best_ms(-1.0), best_ms(2.0)
    assert many > 7500 and few < 200
    assert all_join < 4.0 * none_joins, (all_join, none_joins)


def test_members_of_small_groups_share_their_latencies():
    """Full chip, thousands of members a unit in groups of one or two beside the seed: compaction with all scratch rows joined against none
    (2.2 times; 3.1 when every slot, copied ones too, was handed out by itself)."""
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning8k_b512"].with_(layers=1, kv_heads=1, prefix=200, decode=2800, budget=1536, reserve=768)
    k, v, q = wl.make_unit(w, 0, 0, 0)
    n, T = 240, 3000
    full = lambda x: np.full(n, x, np.int32)
    hb = wl.Batch(wl=w, k=np.tile(k, (n, 1)), v=np.tile(v, (n, 1)), q=np.tile(q[None], (n, 1, 1, 1)), T=full(T), P=full(200), B=full(1536),
                  reserve=full(768), tok_off=np.arange(n + 1, dtype=np.int64) * T, unit_ids=[(i, 0, 0) for i in range(n)])

    def best_us(tau):
        run = gh.GpuRun(hb, tau=tau)
        run.out_struct.rho_core = run.out_struct.rho_rep = run.out_struct.dispersion = None        # (no diagnostics)
        best = np.inf
        for _ in range(8):
            run.ctx.profile_enable(True)
            run.event()
            best = min(best, run.ctx.profile_read()["gather_merge"]["ms"] * 1e3)
            run.ctx.profile_enable(False)
        return best, np.isin(run.out["kind"].cpu().numpy(), (4, 5)).sum() / n

    (joined, many), (none, few) = best_us(-1.0), best_us(2.0)
    assert 1024 < many < 4 * 1536 and few < 1024
    assert joined < 2.65 * none, (joined, none)


@pytest.mark.parametrize("specs,tau,page,dtype", [
    # (rows, prefix, budget, reserve): more slots than the one-kernel compaction has room for, beside shorter units
    ([(14000, 300, 12400, 12200), (1500, 20, 12300, 0), (13000, 12900, 12390, 50)], 0.9, 0, wl.DTYPE_BF16),
    ([(14000, 300, 12400, 12200), (40, 8, 30, 25)], -1.0, 16, wl.DTYPE_FP32),
    # more rows than it counts
    ([(262129, 100, 120, 90), (5000, 10, 60, 55)], 0.9, 0, wl.DTYPE_BF16),
    ([(262200, 261000, 150, 60), (70000, 5, 400, 400)], 0.5, 64, wl.DTYPE_BF16),
])
def test_budgets_and_units_beyond_the_one_kernel_compaction(specs, tau, page, dtype):
    """The event against the staged calls with the same scores, whose selection, weights and status come from kernels of their own."""
    import gpu_harness as gh
    base = wl.WORKLOADS["tiny"].with_(dtype=dtype, head_dim=8, group=2, window=16, cluster_frac=0.6, n_centres=0)
    parts = [wl.make_unit(base.with_(prefix=p, decode=t - p), i, 0, 0) for i, (t, p, b, r) in enumerate(specs)]
    T, P, B, R = (np.array(x, np.int32) for x in zip(*specs))
    hb = wl.Batch(wl=base, k=np.concatenate([p[0] for p in parts]), v=np.concatenate([p[1] for p in parts]),
                  q=np.stack([p[2] for p in parts]), T=T, P=P, B=B, reserve=R,
                  tok_off=np.concatenate([[0], np.cumsum(T)]).astype(np.int64), unit_ids=[(i, 0, 0) for i in range(len(T))])
    run = gh.GpuRun(hb, tau=tau, page_size=page)
    run.ctx.profile_enable(True)
    g = run.event()
    assert run.ctx.device_flags() == 0 and "slot_scan" in run.ctx.profile_read()
    st = gh.GpuRun(hb, tau=tau, page_size=page)
    o, args, ws = st.out, (st.ctx, st.batch, st.prm), (st.ws, st.ws_bytes)
    st.cb.cask_score(*args, o["s"], o["lse"], *ws)
    st.cb.cask_prefix_evict(*args, o["s"], o["kind"], o["plan"], *ws)
    st.cb.cask_select_core(*args, o["s"], o["plan"], o["kind"], *ws)
    st.cb.cask_consolidate_scratch(*args, o["s"], o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"],
                                   o["lost_mass"], *ws)
    st.cb.cask_compact(*args, o["s"], o["kind"], o["seed_of"], o["weight"], st.out_struct, *ws)
    h = st.numpy_outputs()
    merged = 0
    kf, vf = wl.as_float32(hb.k, dtype), wl.as_float32(hb.v, dtype)
    for name in g:
        if name not in ("k_out", "v_out"):
            assert np.array_equal(g[name], h[name]), name
    for u in range(len(specs)):
        a, k = int(hb.tok_off[u]), int(g["n_out"][u])
        assert k == min(int(T[u]), int(B[u]))
        assert np.array_equal(g["k_out"][u][:k], h["k_out"][u][:k]) and np.array_equal(g["v_out"][u][:k], h["v_out"][u][:k])
        # the rows themselves, in 64 bits
        kind, to, wt = (g[x][a:a + int(T[u])] for x in ("kind", "assign", "weight"))
        keep = np.nonzero(np.isin(kind, (1, 2, 3, 4)))[0]
        assert np.array_equal(g["slot_src"][u][:k], keep) and np.array_equal(to[keep], np.arange(k))
        mem = np.nonzero(to >= 0)[0]
        for name, x in (("k_out", kf), ("v_out", vf)):
            want = np.zeros((k, 8))
            np.add.at(want, to[mem], wt[mem, None].astype(np.float64) * x[a + mem])
            tol = 1e-4 * np.abs(want) + 1e-5 if dtype == wl.DTYPE_FP32 else np.maximum(2e-2, np.abs(want) * 2.0 ** -7)
            assert (np.abs(g[name][u][:k] - want) <= tol).all()
        merged += int((kind == 5).sum())
        assert (g["slot_src"][u][k:] == -1).all() and (g["slot_kind"][u][k:] == 0).all() and (g["slot_mass"][u][k:] == 0).all()
    assert merged > 0
