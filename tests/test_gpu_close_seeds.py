"""fp32 scratch rows that are equally close to two seeds, or lie on tau: they go where one fp32 multiply-add after the other, in the order
of the channels, sends them, whatever kernel contracts the keys.  The sums are restated here in numpy: a product of two fp32 numbers
is exact in 64 bits, so adding it to an fp32 number in extended precision and rounding once is a fused multiply-add (but for a
result that lies within 2^-40 of a rounding boundary, which one sum in 10^11 does)."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def fma(a, b, c):
    return (a.astype(np.longdouble) * b + c).astype(np.float32)


def plain_cosines(rows, seeds):
    """[rows, seeds]: dot products channel by channel over the product of the norms."""
    d = rows.shape[1]
    dot = np.zeros((len(rows), len(seeds)), np.float32)
    n = np.zeros((len(rows), 4), np.float32)                       # a row's norm: every fourth channel, added pairwise
    for c in range(d):
        dot = fma(rows[:, c:c + 1], seeds[None, :, c], dot)
        n[:, c % 4] = fma(rows[:, c], rows[:, c], n[:, c % 4])
    nj = np.sqrt((n[:, 0] + n[:, 1]) + (n[:, 2] + n[:, 3]))
    lanes = np.zeros((len(seeds), 32), np.float32)                 # a seed's: every 32nd channel, then pairwise
    for c in range(d):
        lanes[:, c % 32] = fma(seeds[:, c], seeds[:, c], lanes[:, c % 32])
    for off in (16, 8, 4, 2, 1):
        lanes = lanes + lanes[:, np.arange(32) ^ off]
    return dot / (nj[:, None] * np.sqrt(lanes[:, 0])[None, :])


@pytest.mark.parametrize("d,m,page", [(128, 64, 0), (72, 30, 16), (64, 128, 64), (8, 6, 0)])
def test_rows_between_two_seeds(d, m, page):
    import gpu_harness as gh
    rng = np.random.default_rng(d)
    P, W, n_u, T = 40, 16, 2, 1500
    w = wl.WORKLOADS["tiny"].with_(kv_heads=n_u, group=2, window=W, head_dim=d, prefix=P, decode=T - P, budget=P + W + 1 + m,
                                   reserve=W + 1 + m)
    hb = wl.make_batch(w)
    swap = np.arange(d) ^ 1
    seed_at, s = [], np.zeros(n_u * T, np.float32)
    for u in range(n_u):
        # pairs of seeds that are one another's mirror image under a swap of neighbouring channels, and rows that are their own:
        # a row's cosines with the two are equal but for rounding
        k = hb.k[u * T:(u + 1) * T]
        mid = rng.normal(size=(m // 2, d // 2)).astype(np.float32).repeat(2, axis=1) * 3
        a = (mid + 0.3 * rng.normal(size=mid.shape)).astype(np.float32)
        at = P + rng.permutation(T - P - W)
        seeds, core = np.sort(at[:m]), at[m]
        k[seeds] = np.concatenate([a, a[:, swap]])[rng.permutation(m)]
        rest = np.setdiff1d(np.arange(P, T - W), np.append(seeds, core))
        own = mid[rng.integers(0, len(mid), len(rest))]
        k[rest] = own * rng.uniform(0.3, 3, (len(rest), 1)).astype(np.float32)
        k[rest[::7]] += rng.normal(size=(len(rest[::7]), d)).astype(np.float32)         # and some that are not
        su = rng.uniform(0.1, 0.2, T).astype(np.float32)
        su[seeds], su[core], su[:P] = 0.5 + 0.1 * rng.random(m), 0.9, 0.3
        s[u * T:(u + 1) * T] = su
        seed_at.append(seeds)
    cb = gh.GpuRun(hb).cb

    def consolidated(tau):
        run = gh.GpuRun(hb, page_size=page, tau=tau, gamma=0.0)
        o, args = run.out, (run.ctx, run.batch, run.prm)
        sd = run.dev_f32(s)
        cb.cask_prefix_evict(*args, sd, o["kind"], o["plan"], run.ws, run.ws_bytes)
        o["plan"][:, 4], o["plan"][:, 5] = 1, m                    # one core row, m seeds
        cb.cask_select_core(*args, sd, o["plan"], o["kind"], run.ws, run.ws_bytes)
        cb.cask_consolidate_scratch(*args, sd, o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"],
                                    o["lost_mass"], run.ws, run.ws_bytes)
        assert run.ctx.device_flags() == 0
        return run.numpy_outputs()

    g = consolidated(0.5)
    tied = differs = 0
    for u in range(n_u):
        sl = slice(u * T, (u + 1) * T)
        kind, seeds = g["kind"][sl], seed_at[u]
        assert np.array_equal(np.nonzero(kind == 4)[0], seeds)
        rows = np.setdiff1d(np.arange(P, T - W), np.nonzero(np.isin(kind, (3, 4)))[0])
        cos = plain_cosines(hb.k[sl][rows], hb.k[sl][seeds])
        best = cos.argmax(1)                                       # the first among equals
        top = cos[np.arange(len(rows)), best]
        joins = top >= np.float32(0.5)
        assert np.array_equal(kind[rows] == 5, joins)
        assert np.array_equal(g["seed_of"][sl][rows[joins]], seeds[best[joins]])
        assert np.abs(g["sim"][sl][rows] - top).max() <= 1e-6
        second = np.sort(cos, 1)[:, -2]
        tied += int((top - second < 1e-6).sum())
        differs += int(((top > second) & (top - second < 3e-7)).sum())
    assert tied > 500 and differs > 20                             # the case is what it says

    # tau on a row's own cosine: it joins at that value and not at the next one
    sl = slice(0, T)
    rows = np.nonzero(g["kind"][sl] == 5)[0]
    cos = plain_cosines(hb.k[sl][rows], hb.k[sl][seed_at[0]]).max(1)
    for x in (3, len(rows) - 2):
        assert consolidated(float(cos[x]))["kind"][rows[x]] == 5
        assert consolidated(float(np.nextafter(cos[x], np.float32(2))))["kind"][rows[x]] == 0


def test_an_event_agrees_with_the_simt_kernels_on_every_seed():
    """The 8k fp32 shape, consolidated by either path from the same scores: every row at the same seed."""
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning8k_b384"].with_(dtype=wl.DTYPE_FP32, layers=4, kv_heads=2, decode=6000)
    hb = wl.make_batch(w)
    g = gh.GpuRun(hb).event()
    b = gh.GpuRun(hb, score_path=1)                                # the SIMT kernels throughout
    o, args = b.out, (b.ctx, b.batch, b.prm)
    sd = b.dev_f32(g["s"])
    b.cb.cask_prefix_evict(*args, sd, o["kind"], o["plan"], b.ws, b.ws_bytes)
    b.cb.cask_select_core(*args, sd, o["plan"], o["kind"], b.ws, b.ws_bytes)
    b.cb.cask_consolidate_scratch(*args, sd, o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"], o["lost_mass"],
                                  b.ws, b.ws_bytes)
    h = b.numpy_outputs()
    for name in ("kind", "seed_of", "lost_mass", "unit_status"):
        assert np.array_equal(g[name], h[name]), name
    assert np.abs(g["sim"] - h["sim"]).max() <= 1e-6
