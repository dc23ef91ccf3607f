"""Tensor-core scoring over query-row counts and head dims: every division of the rows into blocks and row groups, against
the oracle.  Scores are checked to 1e-5 relative inside compare_event (the bound of the other parity tests: means of
exponentials whose fp32 arguments are off by a few units in the last place)."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,window,d,page,tail", [
    (1, 33, 128, 0, 5),       # one block of 128 rows, four key tiles a step; rows not a multiple of 32
    (1, 128, 64, 16, 300),    # a full block, one 64-channel half, paged
    (1, 130, 128, 0, 70),     # two blocks, the second with two rows
    (2, 128, 80, 0, 1),       # two full blocks, two tiles a step, a zero-padded head dim
    (5, 48, 96, 64, 40),      # 240 rows: a half-filled last block
    (3, 100, 128, 0, 127),    # 300 rows: four slots, one of them unused
    (7, 64, 128, 0, 50),      # 448 rows: the fourth block half filled
    (5, 78, 128, 64, 9),      # 390 rows: six of its rows, window not a multiple of 16
    (2, 130, 128, 16, 100),   # 260 rows: the third block half filled, no fourth
    (3, 128, 96, 0, 64),      # 384 rows: three whole blocks
    (7, 64, 96, 16, 90),      # 448 rows below head_dim 113: the general form of the kernels
    (3, 100, 64, 0, 31),      # 300 rows there
    (10, 48, 128, 0, 61),     # 480 rows, a block of 32 columns in two heads
    (13, 60, 128, 64, 77),    # 780 rows: two row groups of 416 and 364, the fourth block a quarter filled and empty
    (14, 64, 128, 0, 99),     # 896 rows: two row groups of 448
    (15, 60, 128, 0, 20),     # 900 rows: two row groups of 480 and 420
    (7, 96, 72, 0, 33),       # 672 rows: three row groups of two blocks
    (8, 128, 128, 0, 77),     # 1,024 rows: two row groups of four blocks
    (9, 128, 128, 128, 10),   # 1,152 rows: five row groups, the last one short
    (8, 128, 8, 0, 3),        # the narrowest head
])
def test_query_rows_and_head_dims(group, window, d, page, tail):
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning32k_b512"].with_(layers=1, kv_heads=3, group=group, window=window, head_dim=d, prefix=201,
                                                 decode=1024 + tail, budget=384, reserve=192)
    hb = wl.make_batch(w)
    run = gh.GpuRun(hb, page_size=page)
    g = run.event()
    assert run.ctx.used_tensor_path and run.ctx.device_flags() == 0
    st = gh.compare_event(hb, g, gh.run_oracle(hb))
    assert st["max_score_rel"] < 1e-5 and st["cascaded"] <= 1


@pytest.mark.parametrize("group,window", [(1, 64), (4, 64), (8, 128)])
def test_row_groups_with_supplied_normalisers_and_many_units(group, window):
    """More units than multiprocessors, of one to eleven tiles each, so that segments begin and end anywhere in a step;
    with the normalisers of the oracle the score pass runs alone."""
    import gpu_harness as gh
    from oracle import cask_oracle as orc
    rng = np.random.default_rng(group)
    base = wl.WORKLOADS["serving_steady_b512"].with_(layers=1, kv_heads=1, group=group, window=window, carried_rows=0)
    parts, T = [], []
    for i in range(200):
        t = int(rng.integers(window, 1400))
        parts.append(wl.make_unit(base.with_(prefix=t // 3, decode=t - t // 3), i, 0, 0))
        T.append(t)
    tok = np.concatenate([[0], np.cumsum(T)]).astype(np.int64)
    T = np.array(T, np.int32)
    n = len(T)
    hb = wl.Batch(wl=base, k=np.concatenate([p[0] for p in parts]), v=np.concatenate([p[1] for p in parts]),
                  q=np.stack([p[2] for p in parts]), T=T, P=T // 3, B=np.full(n, 128, np.int32),
                  reserve=np.full(n, 64, np.int32), tok_off=tok, unit_ids=[(i, 0, 0) for i in range(n)])
    want, lse = orc.score_batch(wl.as_float32(hb.k, 0), wl.as_float32(hb.q, 0), tok)
    for lse_in in (None, lse.reshape(n, -1)):
        run = gh.GpuRun(hb, lse_in=lse_in)
        g = run.event()
        assert run.ctx.used_tensor_path and run.ctx.device_flags() == 0
        big = want > 1e-12
        assert (np.abs(g["s"][big] - want[big]) <= 1e-5 * want[big]).all()
        assert np.abs(g["s"][~big] - want[~big]).max(initial=0.0) <= 1e-12


@pytest.mark.parametrize("group,window,d,page,tail,budget", [
    (1, 32, 8, 0, 0, 96),           # the narrowest head, one row block, whole tiles
    (2, 16, 64, 48, 5, 128),        # one 64-channel half, pages that do not divide a tile
    (4, 33, 72, 0, 127, 384),       # two row groups of unequal length, a zero-padded head dim
    (7, 64, 128, 16, 1, 512),       # four row groups; m = 96 seeds
    (1, 100, 128, 0, 60, 800),      # m = 128 seeds: every seed column in use
    (8, 128, 96, 0, 33, 1000),      # eight row groups; more than 128 seeds: SIMT assignment beside the split scoring
])
def test_fp32_caches_through_their_bf16_parts(group, window, d, page, tail, budget):
    """fp32 events on the tensor cores keep fp32 accuracy: scores within 2e-6 of the oracle (the six part products are exact
    to 2^-26 and the additions round as fp32 ones do; the SIMT kernel is held to 1e-5), merged rows within 1e-4, and twice the
    same bytes; the SIMT kernels agree."""
    import gpu_harness as gh
    w = wl.WORKLOADS["tiny"].with_(kv_heads=3, group=group, window=window, head_dim=d, prefix=77, decode=1152 + tail,
                                   budget=budget, reserve=budget - 60, cluster_frac=0.6, n_centres=0)
    hb = wl.make_batch(w)
    run = gh.GpuRun(hb, page_size=page)
    names = {run.ctx._lib.cask_kernel_name(i).decode() for i in range(run.ctx._lib.cask_kernel_count())}
    assert "split_rows" in names
    run.ctx.profile_enable(True)
    g = run.event()
    assert run.ctx.profile_read()["split_rows"]["launches"] == 1 and run.ctx.device_flags() == 0
    run.ctx.profile_enable(False)
    st = gh.compare_event(hb, g, gh.run_oracle(hb))
    assert st["max_score_rel"] < 2e-6 and st["cascaded"] <= 1
    again = gh.GpuRun(hb, page_size=page).event()
    for name in g:
        assert np.array_equal(g[name], again[name]), name
    simt = gh.GpuRun(hb, page_size=page, score_path=1).event()
    big = simt["s"] > 1e-12
    assert (np.abs(g["s"] - simt["s"])[big] <= 1e-5 * simt["s"][big]).all()



@pytest.mark.parametrize("dtype,d,score_path,want", [(wl.DTYPE_BF16, 128, 0, 1), (wl.DTYPE_FP32, 128, 0, 2), (wl.DTYPE_FP32, 64, 0, 2),
                                                    (wl.DTYPE_FP32, 128, 1, 0), (wl.DTYPE_FP32, 200, 0, 0), (wl.DTYPE_BF16, 128, 1, 0)])
def test_the_path_that_scored_is_told(dtype, d, score_path, want):
    """The kernels that ran, and the clocks of the tensor-core passes wherever those ran."""
    import gpu_harness as gh
    w = wl.WORKLOADS["tiny"].with_(dtype=dtype, head_dim=d, decode=3000)
    run = gh.GpuRun(wl.make_batch(w), score_path=score_path)
    run.event()
    assert run.ctx.score_path == want and run.ctx.used_tensor_path == (want == 1)
    clocks = run.ctx.score_clock_mhz()
    assert all(c > 100.0 for c in clocks) if want else clocks == (0.0, 0.0)


def test_fp32_numbers_above_the_greatest_bf16_number():
    """Keys of up to 3.4e38, which bf16 would round to infinity, against queries that make ordinary logits of them."""
    import gpu_harness as gh
    from oracle import cask_oracle as orc
    hb = wl.make_batch(wl.WORKLOADS["tiny"].with_(decode=1500))
    rng = np.random.default_rng(0)
    big = rng.permutation(len(hb.k))[:300]
    hb.k[:, 5] = 0.0
    hb.k[big, 5] = (rng.uniform(3.38, 3.4028234e38 / 1e38, len(big)) * 1e38 * rng.choice([-1, 1], len(big))).astype(np.float32)
    assert (np.abs(hb.k[big, 5]) > 3.3961e38).any()               # beyond the last number that rounds to a finite bf16
    hb.q[..., 5] = np.float32(2.0 ** -126) * rng.choice([1, 2, 4], hb.q.shape[:-1]).astype(np.float32)
    run = gh.GpuRun(hb)
    run.cb.cask_score(run.ctx, run.batch, run.prm, run.out["s"], run.out["lse"], run.ws, run.ws_bytes)
    s = run.out["s"].cpu().numpy()
    assert run.ctx.score_path == 2
    want, _ = orc.score_batch(hb.k, hb.q, hb.tok_off)
    assert (np.abs(s - want) <= 1e-5 * want + 1e-12).all()
