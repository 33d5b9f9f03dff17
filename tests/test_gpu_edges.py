"""Edge sizes of kernels whose dispatch or layout depends on sizes, against the oracle.

All outputs are integers: the bar is equality.
"""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import assert_rows_equal, need_gpu, rec_rows, run_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    c = binding.Context(0)
    yield c
    c.close()


def to_dev(a):
    torch = need_gpu()
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def tandem_genome(seed, unit_lo=60, unit_hi=1500):
    """Duplications whose insides hold tandem units of many lengths: target
    hashes recur at distances around a window's span, inside one warp's 32
    records and across them."""
    rng = np.random.default_rng(seed)
    seq = synth.random_bases(rng, 90_000, 0.45)
    at = 3_000
    for u in np.geomspace(unit_lo, unit_hi, 7).astype(int):
        unit = synth.random_bases(rng, int(u), 0.45)
        arr = np.tile(unit, max(2, 2600 // int(u)))[:3000]
        arr = synth.mutate(rng, arr, 0.985)
        seq[at:at + len(arr)] = arr
        copy = synth.mutate(rng, seq[at - 300:at + len(arr) + 300], 0.93)
        if rng.random() < 0.5:
            copy = synth.reverse_complement(copy)
        dst = at + 45_000
        seq[dst:dst + len(copy)] = copy
        at += 5_500
    return synth.genome_from_parts([seq])


@pytest.mark.parametrize("pd", [
    dict(), dict(w=50), dict(w=10), dict(w=7, query_step=100),  # 64, 192, 256 counters a roll
    dict(w=24, n=300, query_step=75), dict(k=11, w=16, max_occ=40), dict(k=14, w=12)])
def test_refine_recurring_hashes(ctx, pd):
    pd = dict(pd)
    step = pd.pop("query_step", 250)
    d = oracle.params(**pd)
    d["step"] = step
    g = tandem_genome(4)
    recs = oracle.sketch(g.seq, g.offsets, d)
    want = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d)
    p = binding.params_from_dict(d)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    assert_rows_equal(rec_rows(rec), recs, "sketch")
    srt, off = ctx.sedef_index(rec, p)
    runs, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert n > 20
    assert_rows_equal(run_rows(runs), want, "runs")
