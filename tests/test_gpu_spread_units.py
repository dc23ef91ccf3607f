"""Few long units: every unit's normaliser partials come from many CTAs, and a CTA on the border of two units makes both row tables
at its start.  Scores of the tensor-core passes against the SIMT ones."""
import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("units,decode,group,window", [
    (5, 5000, 4, 128),          # four blocks a tile; 30 CTAs a unit, most borders inside one
    (3, 9001, 7, 64),           # 448 rows
    (5, 5000, 4, 64),           # two blocks a tile
    (33, 2000, 8, 64),          # just above four CTAs a unit
    (40, 2000, 8, 64),          # and below
])
def test_scores_of_few_long_units(units, decode, group, window):
    import gpu_harness as gh
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=group, window=window, prefix=100, decode=decode,
                                                budget=400, reserve=200)
    hb = wl.make_batch(w)
    run = gh.GpuRun(hb)
    got = run.event()
    assert run.ctx.device_flags() == 0 and run.ctx.used_tensor_path
    want = gh.GpuRun(hb, score_path=1).event()
    # both sums are exact to some 1e-6: products of bf16 in fp32, exponentials to 2^-22
    assert np.allclose(got["s"], want["s"], rtol=gh.SCORE_RTOL, atol=1e-12)
    for u in range(units):
        a = int(hb.tok_off[u])
        assert abs(float(got["s"][a:a + int(hb.T[u])].sum()) - 1.0) < 1e-4


def _kernel_us(hb, name, **kw):
    """Shortest of eight profiled times of one kernel of the event, and the event's normalisers."""
    import gpu_harness as gh
    run = gh.GpuRun(hb, **kw)
    run.out_struct.rho_core = run.out_struct.rho_rep = run.out_struct.dispersion = None        # (no diagnostics)
    best = np.inf
    for _ in range(8):
        run.ctx.profile_enable(True)
        g = run.event()
        best = min(best, run.ctx.profile_read()[name]["ms"] * 1e3)
        run.ctx.profile_enable(False)
    return best, g["lse"]


def test_a_rows_partials_are_walked_once():
    """One unit on all CTAs has two partials a CTA and row, and their fold is most of the score pass: three times what the pass takes
    with given normalisers, which has none (five times when a trial run of the table's code went over as many again)."""
    hb = wl.make_batch(wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=1, group=4, window=128, prefix=100, decode=18800, budget=512,
                                                              reserve=256))
    own, lse = _kernel_us(hb, "score_mass")
    given, _ = _kernel_us(hb, "score_mass", lse_in=lse)
    assert own < 4.0 * given, (own, given)
