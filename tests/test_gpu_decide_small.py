"""The event's one-kernel selection and seed gather of short units against the staged calls (counting or radix selection, one
kernel per step): the same scores go in, everything must come out the same, byte for byte."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

BF16, FP32 = wl.DTYPE_BF16, wl.DTYPE_FP32
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefix,decode,budget,reserve,dup,page,dtype,head_dim", [
    (0, 65, 40, 40, 0, 0, BF16, 128),            # no prefix, the shortest scratch range
    (960, 64, 300, 120, 0, 0, BF16, 128),        # 1,024 rows, nearly all of them prefix
    (0, 1024, 700, 700, 0, 16, BF16, 128),       # 1,024 rows, all of them decode; more seeds than a block has threads
    (256, 384, 512, 256, 0, 1, BF16, 128),       # a page per row
    (100, 900, 400, 390, 1, 0, BF16, 128),       # every decode key the same: one bin holds the whole range
    (500, 500, 300, 200, 1, 16, BF16, 128),      # and every prefix key too
    (64, 800, 300, 236, 3, 0, BF16, 128),        # three distinct decode keys
    (300, 400, 360, 60, 0, 0, BF16, 128),        # decode budget of the recent rows alone
    (300, 700, 950, 650, 0, 0, FP32, 64),        # nearly all rows kept; seeds as three parts
    (130, 300, 200, 150, 0, 16, BF16, 256),      # two rounds of channels
    (130, 300, 200, 150, 2, 0, FP32, 72),        # a last round that not all lanes have
])
def test_short_units_equal_the_staged_calls(prefix, decode, budget, reserve, dup, page, dtype, head_dim):
    import gpu_harness as gh
    import torch
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=3, group=2, window=32, prefix=prefix, decode=decode, budget=budget,
                                                reserve=reserve, dtype=dtype, head_dim=head_dim)
    hb = wl.make_batch(w)
    if dup:
        for u in range(hb.n_units):
            a = int(hb.tok_off[u])
            if prefix == decode:
                hb.k[a:a + prefix] = hb.k[a]
            hb.k[a + prefix:a + prefix + decode] = hb.k[a + prefix + np.arange(decode) % dup]
    run = gh.GpuRun(hb, page_size=page)
    g = run.event()
    assert run.ctx.device_flags() == 0
    st = gh.GpuRun(hb, page_size=page)
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


@pytest.mark.parametrize("prefix,decode,budget,reserve,dup,page,dtype,head_dim", [
    (0, 65, 40, 40, 0, 0, BF16, 128),
    (0, 1024, 700, 700, 0, 16, BF16, 128),       # 1,024 rows, several rounds of seeds
    (500, 500, 300, 200, 1, 16, BF16, 128),      # a bin with every prefix row, one with every decode row
    (212, 300, 400, 250, 0, 0, FP32, 64),        # 512 rows
    (213, 300, 400, 250, 0, 1, BF16, 256),       # one more, a page per row
])
def test_threads_by_the_number_of_units(prefix, decode, budget, reserve, dup, page, dtype, head_dim):
    """The selection of a short unit runs with 256 to 1,024 threads, by how many units there are: three units alone, and copies of them in
    batches of more than one and more than three units a multiprocessor.  The normalisers are given and the 512 query rows fill a tile's four
    slots (the fp32 units are a single step of tiles), so that a unit's scores do not depend on the batch."""
    import gpu_harness as gh
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=3, group=16, window=32, prefix=prefix, decode=decode, budget=budget,
                                                reserve=reserve, dtype=dtype, head_dim=head_dim)
    one = wl.make_batch(w)
    if dup:
        one.k[:] = one.k[0]
    T = prefix + decode
    lse = np.random.default_rng(1).uniform(5.0, 9.0, (3, 512)).astype(np.float32)

    def event(copies):
        n = 3 * copies
        full = lambda x: np.full(n, x, np.int32)
        hb = wl.Batch(wl=w, k=np.tile(one.k, (copies, 1)), v=np.tile(one.v, (copies, 1)), q=np.tile(one.q, (copies, 1, 1, 1)), T=full(T), P=full(prefix),
                      B=full(budget), reserve=full(reserve), tok_off=np.arange(n + 1, dtype=np.int64) * T, unit_ids=[(i, 0, 0) for i in range(n)])
        run = gh.GpuRun(hb, page_size=page, lse_in=np.tile(lse, (copies, 1)))
        g = run.event()
        assert run.ctx.device_flags() == 0
        return {name: x.reshape(copies, -1) for name, x in g.items()}

    want = event(1)
    for copies in (sms // 3 + 2, sms + 2):
        for name, x in event(copies).items():
            if name in ("k_out", "v_out"):
                x, y = x.reshape(3 * copies, budget, -1), want[name].reshape(3, budget, -1)
                for u in range(3 * copies):
                    k = int(want["n_out"][0][u % 3])
                    assert np.array_equal(x[u][:k], y[u % 3][:k]), name
            else:
                assert (x.view(np.uint8) == want[name].view(np.uint8)).all(), name
