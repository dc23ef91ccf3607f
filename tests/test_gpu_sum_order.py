"""The order in which the terms of a score are added is kept from one version to the next: two rows whose scores agree to 1e-7 at a
selection boundary, or two seeds whose cosines with a row do, are told apart by it, and a changed order hands slots to other rows.

The digests in golden/sum_order.json are those of the library before its scoring passes served more than 512 query rows, taken on a
B200 (148 multiprocessors: the normalisers of a unit are added up by the CTAs that share its tiles).  A digest changes with any
change of a rounding; what is compared is the 32-bit patterns."""
import hashlib
import json
import os

import numpy as np
import pytest

from paper_2604_10900_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = {     # group, window, rows of the prefix, of the decode region, units, page size, causal, normalisers given
    "rows448": (7, 64, 200, 1500, 6, 0, 1, False),                 # the fourth block half filled
    "rows448_paged": (7, 64, 256, 3001, 4, 16, 1, True),
    "rows416": (13, 32, 77, 1033, 3, 0, 1, False),                 # a quarter of it
    "rows512": (4, 128, 256, 384, 200, 16, 1, False),              # short units, one tile of five on the causal diagonal
    "rows512_long": (8, 64, 512, 20007, 2, 0, 1, False),           # a unit's tiles spread over many CTAs
    "rows512_all_visible": (4, 128, 100, 1177, 5, 64, 0, True),    # no causal mask: the ragged tile alone is masked
}


def event(name):
    import gpu_harness as gh
    group, window, prefix, decode, units, page, causal, given = CASES[name]
    w = wl.WORKLOADS["reasoning8k_b384"].with_(layers=1, kv_heads=units, group=group, window=window, prefix=prefix, decode=decode)
    hb = wl.make_batch(w)
    lse = None
    if given:      # any numbers of a plausible size serve here
        lse = np.random.default_rng(3).uniform(7.0, 12.0, (hb.n_units, group * window)).astype(np.float32)
    return gh.GpuRun(hb, page_size=page, causal=causal, lse_in=lse).event()


def digest(a):
    return hashlib.sha256(np.ascontiguousarray(a).tobytes()).hexdigest()[:32]


def golden(name):
    with open(os.path.join(os.path.dirname(__file__), "golden", "sum_order.json")) as f:
        return json.load(f)[name]


@pytest.mark.parametrize("name", CASES)
def test_scores_and_normalisers(name):
    g, want = event(name), golden(name)
    assert digest(g["lse"]) == want["lse"]
    assert digest(g["s"]) == want["s"]
    for out in ("kind", "slot_src", "lost_mass"):
        assert digest(g[out]) == want[out], out


@pytest.mark.parametrize("name", CASES)
def test_cosines(name):
    """Best cosine of every scratch row and the seed it belongs to, norms of rows and seeds included."""
    g, want = event(name), golden(name)
    assert digest(g["seed_of"]) == want["seed_of"]
    assert digest(g["sim"]) == want["sim"]
