"""More than 256 seeds a unit: the tensor-core assignment takes them in chunks, a launch each, and leaves the rows its sums cannot tell to a
kernel with the SIMT kernel's sums.  The SIMT kernel, which served these shapes before, is the reference: the same scores and selections
go in, and every row has to go where that kernel sends it."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _compare(hb, page=0, change=None, **kw):
    import gpu_harness as gh
    import torch
    tc, simt = (gh.GpuRun(hb, page_size=page, **kw) for _ in range(2))
    if change:
        for run in (tc, simt):
            change(run)
    slow = simt.cb.params(score_path=1, **kw)
    outs = []
    for run, prm in ((tc, tc.prm), (simt, slow)):
        o, args = run.out, (run.ctx, run.batch)
        ws = (run.ws, run.ws_bytes)
        run.cb.cask_score(*args, run.prm, o["s"], o["lse"], *ws)
        run.cb.cask_prefix_evict(*args, run.prm, o["s"], o["kind"], o["plan"], *ws)
        run.cb.cask_select_core(*args, run.prm, o["s"], o["plan"], o["kind"], *ws)
        run.cb.cask_consolidate_scratch(*args, prm, o["s"], o["plan"], o["kind"], o["seed_of"], o["weight"], o["sim"], o["unit_status"], o["lost_mass"], *ws)
        torch.cuda.synchronize()
        assert run.ctx.device_flags() == 0
        outs.append({n: o[n].cpu().numpy() for n in ("s", "kind", "seed_of", "weight", "unit_status", "lost_mass", "sim", "plan")})
    a, b = outs
    for name in a:
        if name == "sim":      # both are sums of 128 products of at most the norms' product: off by up to 128 roundings of 2^-24 each
            assert np.abs(a["sim"] - b["sim"]).max() <= 2 * 128 * 2.0 ** -24
        else:
            assert np.array_equal(a[name].view(np.uint8), b[name].view(np.uint8)), name
    if page == 0 and not change:
        ev = gh.GpuRun(hb, **kw)
        e = ev.event()
        for name in ("kind", "seed_of", "lost_mass"):
            assert np.array_equal(e[name].view(np.uint8), a[name].view(np.uint8)), name
    return a


def _batch(units=3, prefix=100, decode=1500, budget=800, reserve=700, head_dim=128, window=32):
    return wl.make_batch(wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=4, window=window, prefix=prefix, decode=decode,
                                                                budget=budget, reserve=reserve, head_dim=head_dim))


@pytest.mark.parametrize("m,kw,page", [
    (257, dict(), 0),                                      # three chunks of 96, the last of 65
    (288, dict(units=5), 16),                              # three whole chunks
    (385, dict(decode=1283), 0),                           # four chunks, the last of 73; a ragged last tile
    (700, dict(head_dim=64, decode=2001), 0),
    (300, dict(head_dim=72, units=160, decode=700), 64),   # more units than multiprocessors
    (1100, dict(units=2, decode=2600), 0),                 # more seeds than a selection's list holds
    (284, dict(units=2, decode=17000, budget=652, reserve=600, window=32), 0),      # long units: listed slots and rows that join
])
def test_rows_go_where_the_simt_kernel_sends_them(m, kw, page):
    kw = dict(kw)
    if "budget" not in kw:     # room for r recent rows, m - 1 or m core rows and m seeds beside a prefix of 100 rows
        kw.update(budget=100 + 32 + 2 * m, reserve=32 + 2 * m)
    a = _compare(_batch(**kw), page)
    assert (a["plan"][:, 5] == m).all(), a["plan"][:, 5]
    assert (a["kind"] == 5).any() and (a["kind"] == 0).any()


@pytest.mark.parametrize("tau", [-1.0, 0.3])
def test_thresholds(tau):
    _compare(_batch(), tau=tau)


def test_units_of_few_and_many_seeds():
    """Budgets from a handful of seeds to several chunks: a unit is finished by the launch with its last chunk and passed over by the rest."""
    hb = _batch(units=12)
    hb.B[:] = [800, 60, 400, 1100, 100, 800, 140, 700, 220, 1500, 70, 360]
    hb.reserve[:] = np.maximum(hb.B - 100, 40)
    a = _compare(hb)
    assert a["plan"][:, 5].min() < 16 and a["plan"][:, 5].max() > 600


def test_equal_and_empty_rows():
    """Seeds equal to one another, rows equal to seeds, rows and seeds of zeros, rows with a number that is none: nothing is certain, and
    the first seed among equals wins."""
    hb = _batch(units=2, decode=900)
    rng = np.random.default_rng(3)
    T = int(hb.T[0])
    k = hb.k.reshape(2, T, -1)
    k[0, 100:] = k[0, 100 + rng.integers(0, 5, T - 100)]          # five distinct keys
    k[1, rng.permutation(np.arange(100, T))[:300]] = 0

    def nan_row(run):
        run.dev["k"].view(2, T, -1)[1, 700] = float("nan")
    _compare(hb)
    _compare(hb, change=nan_row)


@pytest.mark.parametrize("units,head_dim,distinct,decode,budget,page", [
    (12, 128, 40, 1500, 800, 0),         # runs of rows from the list
    (160, 128, 300, 900, 700, 0),
    (24, 72, 1000, 1500, 800, 0),
    (12, 128, 40, 3000, 750, 0),         # more than half of all rows: tile by tile
    (5, 80, 30, 3011, 750, 64),
])
def test_more_uncertain_rows_than_there_are_blocks(units, head_dim, distinct, decode, budget, page):
    """Nearly every row repeats: several rows of a unit are decided at a time, in runs that end where the list goes on with another unit, or
    whole tiles."""
    hb = _batch(units=units, head_dim=head_dim, decode=decode, budget=budget, reserve=budget - 50 if decode < 1000 else 700)
    T = int(hb.T[0])
    k = hb.k.reshape(units, T, -1)
    rng = np.random.default_rng(units)
    for u in range(units):
        k[u, 100:] = k[u, 100 + rng.integers(0, distinct, T - 100)]
    a = _compare(hb, page)
    assert a["plan"][:, 5].min() > 256


def _no_seeds(run):
    run.ws.fill_(0x7f)      # what a workspace held before is no value, seed or row of this call


@pytest.mark.parametrize("kw,page", [(dict(), 0), (dict(budget=1400, reserve=1300), 16), (dict(units=160, decode=900, budget=700, reserve=650, head_dim=64), 0)])
def test_a_workspace_full_of_numbers_that_are_no_seeds(kw, page):
    _compare(_batch(**kw), page, change=_no_seeds)


def test_near_seeds_whose_plain_sums_round_apart(monkeypatch):
    """A row of cosines 1.28e-5 apart with two seeds, the products with one rounded up at every addition of the plain sum and those with the
    other lost: the plain sums order the seeds the other way round than the cosines, by 1.4e-6."""
    hb = _batch(units=2)
    T, eps = int(hb.T[0]), 2.0 ** -12

    def key(x, rest):
        v = np.zeros(128, np.float32)
        v[0], v[1:121], v[121:] = 1, x, rest
        u = v.view(np.uint32)
        return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)
    row, rounded, lost = key(eps, 0), key(eps * (1 + 2.0 ** -7), (1.28e-5 / 3.5) ** 0.5), key(eps * (1 - 2.0 ** -8), 0)
    k = hb.k.reshape(2, T, -1)
    k[:, 900:1300] = row
    k[0, 500], k[0, 600] = rounded, lost            # among the seeds, decode rows 334 to 667 in the order of the scores
    k[1, 500], k[1, 600] = lost, rounded
    import torch
    from paper_2604_10900_b200 import binding as cb
    scores = torch.from_numpy(np.tile(np.linspace(1, 0.1, T, dtype=np.float32), 2))
    monkeypatch.setattr(cb, "cask_score", lambda ctx, batch, prm, s, *rest: s.copy_(scores))
    a = _compare(hb, change=_no_seeds)
    assert (a["seed_of"].reshape(2, T)[0, 900:1300] == 500).all() and (a["seed_of"].reshape(2, T)[1, 900:1300] == 600).all()


@pytest.mark.parametrize("units,head_dim,distinct,decode,page", [
    (12, 128, 40, 3000, 0),          # 64 channels at a time
    (5, 72, 30, 3011, 64),           # all 72 at a time; a ragged last tile
    (4, 80, 60, 2000, 0),
    (3, 120, 25, 1283, 16),          # 64 and 56
    (3, 8, 20, 1283, 0),             # one piece of a row
])
def test_caches_that_repeat_and_a_threshold_that_every_row_passes(units, head_dim, distinct, decode, page):
    """At tau = -1 every row is as near to a seed as to its copies, so more than a quarter of all rows are listed and go tile by tile."""
    hb = _batch(units=units, head_dim=head_dim, decode=decode, budget=750)
    T = int(hb.T[0])
    k = hb.k.reshape(units, T, -1)
    rng = np.random.default_rng(units)
    for u in range(units):
        k[u, 100:] = k[u, 100 + rng.integers(0, distinct, T - 100)]
    a = _compare(hb, page, tau=-1.0)
    assert a["plan"][:, 5].min() > 256 and (a["kind"] == 5).mean() > 0.25


@pytest.mark.parametrize("head_dim,page,kw,tau", [
    (128, 0, dict(), 0.9),                                             # 334 seeds, three chunks
    (64, 16, dict(decode=2001, budget=900), 0.3),                      # most rows join
    (128, 0, dict(decode=6000, budget=652, reserve=600), 0.9),         # longer units: listed slots and rows that join
])
def test_events_with_carried_masses_against_the_oracle(head_dim, page, kw, tau):
    """The whole event, compacted rows and all, and the chunks' launches: this is not the SIMT kernel's path."""
    import gpu_harness as gh
    hb = _batch(units=2, head_dim=head_dim, **kw)
    hb.mass_in = np.random.default_rng(head_dim).uniform(0, 2e-3, int(hb.tok_off[-1])).astype(np.float32)
    run = gh.GpuRun(hb, page_size=page, tau=tau)
    run.ctx.profile_enable(True)
    g = run.event()
    m = int(g["plan"][:, 5].max())
    assert m > 256 and run.ctx.profile_read()["assign"]["launches"] == -(-m // 128) + 1 and run.ctx.device_flags() == 0
    st = gh.compare_event(hb, g, gh.run_oracle(hb, tau=tau), tau=tau)
    assert st["merged_elems"] > 0 and (g["kind"] == 5).any()


@pytest.mark.parametrize("distinct", [0, 40])
def test_a_host_resident_cache_gives_the_device_events_bytes(distinct):
    """The list of close rows is emptied by another route there; with rows that repeat it is long, in both of two calls."""
    import gpu_harness as gh
    import torch
    hb = _batch(units=3)
    if distinct:
        k, rng = hb.k.reshape(3, int(hb.T[0]), -1), np.random.default_rng(distinct)
        for u in range(3):
            k[u, 100:] = k[u, 100 + rng.integers(0, distinct, 1500)]
    w, run = hb.wl, gh.GpuRun(hb, tau=0.3)
    run.event()
    cb = run.cb
    batch, keep = cb.make_batch(hb.k, hb.v, hb.q, hb.T, hb.P, hb.B, hb.reserve, hb.tok_off, w.head_dim, w.group, w.window, w.dtype)
    nbytes = cb.cask_host_event_device_bytes(batch, run.prm, run.Bmax)
    dev = torch.full((nbytes,), 0x7f, dtype=torch.uint8, device="cuda:0")
    want = {name: t.cpu().view(torch.uint8).numpy() for name, t in run.out.items()}
    ho = {name: np.zeros(t.cpu().view(torch.uint8).shape, np.uint8) for name, t in run.out.items()}
    for _ in range(2):
        cb.cask_compress_event_host(run.ctx, batch, run.prm, cb.make_outputs(ho, run.Bmax), dev, nbytes)
    assert run.ctx.device_flags() == 0 and (run.out["n_out"].cpu().numpy() == hb.B).all()
    for name in want:
        assert np.array_equal(ho[name], want[name]), name
