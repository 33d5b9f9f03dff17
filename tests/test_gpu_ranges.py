"""Where the posting ranges of a self-search pay, and that the runs are the same either way."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import assert_rows_equal, need_gpu, run_rows
from tests.test_gpu_edges import crowded_genome, tandem_genome

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    c = binding.Context(0)
    c.sedef_trace_enable(True)
    yield c
    c.close()


def to_dev(a):
    return need_gpu().from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def filtered(ctx, rec, srt, off, offsets, p):
    """Runs, and whether the records' ranges were looked up."""
    ctx.sedef_trace_report(reset=True)
    runs, _ = ctx.sedef_filter(rec, offsets, rec, srt, off, offsets, p)
    return run_rows(runs), any(x.endswith("k_qpost") for x in ctx.sedef_trace_report(reset=True))


# steps at which the ranges pay and do not, through every tier (families of copies of many sizes)
@pytest.mark.parametrize("pd,step,taken", [
    (dict(), 7, True), (dict(), 250, False), (dict(self_mode=2), 7, True), (dict(self_mode=2), 250, False),
    (dict(k=14), 7, True), (dict(k=9, w=20), 6, True), (dict(w=40), 3, True), (dict(max_occ=30), 7, True),
    (dict(delta_m=0.9, delta_g=0.2, w=60), 4, False), (dict(w=4), 30, False)])
def test_runs_with_and_without_ranges(ctx, pd, step, taken):
    d = oracle.params(**pd)
    d["step"] = step
    g = crowded_genome(12) if pd.get("w") != 4 else tandem_genome(3)
    recs = oracle.sketch(g.seq, g.offsets, d)
    p = binding.params_from_dict(d)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    got, looked_up = filtered(ctx, rec, srt, off, g.offsets, p)
    assert looked_up == taken
    some = dict(d, step=12 * step)  # the oracle on every twelfth window of each sequence
    start = g.offsets[np.searchsorted(g.offsets, got[:, 0], side="right") - 1]
    want = oracle.filter_runs(recs, g.offsets, recs, g.offsets, some, threads=16)
    assert_rows_equal(got[(got[:, 0] - start) % (12 * step) == 0], want, "runs")
    assert len(want) > 20
    if taken:
        assert_rows_equal(run_rows(ctx.selfsearch_graph(to_dev(g.seq), g.offsets, p).outputs()["runs"]), got,
                          "captured runs")


def test_few_windows_of_many_records(ctx):
    """A few windows do not pay for a walk over all records."""
    s = np.empty(30_000_000, dtype=np.uint8)
    synth.random_bases_chunked(np.random.default_rng(4), s, 0.45)
    for parts, mode in ((1, 1), (300, 2)):
        off_seq = np.linspace(0, len(s), parts + 1).astype(np.int64)
        p = binding.params(self_mode=mode)
        rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(s)), off_seq, p)
        srt, off = ctx.sedef_index(rec, p)
        for step, taken in ((250, True), (20_000, False), (5_000_000, False)):
            p.query_step = step
            assert filtered(ctx, rec, srt, off, off_seq, p)[1] == taken, (mode, step)
