"""The autotuner on query records that are not the index's own (a sample of them, a copy)."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import assert_rows_equal, need_gpu, run_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("which", ["half", "head", "copy"])
def test_autotune_on_other_records(mode, which):
    """Posting ranges by a walk over the index need its own records in the query: a target record
    past the query's last one has a rank past the array.  Others are searched one by one."""
    torch = need_gpu()
    ctx = binding.Context(0)
    g = synth.small_case(31, lengths=(120_000, 60_000), n_sd=8, sd_lo=1500, sd_hi=6000, mask_frac=0.1)
    d = oracle.params(self_mode=mode)
    d["step"] = 3  # many windows: the ranges pay
    p = binding.params_from_dict(d)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(torch.from_numpy(g.seq).to("cuda:0")), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    n = rec.numel() // 64 * 64
    query = {"half": rec[::2].clone(), "head": rec[:n].clone(), "copy": rec.clone()}[which]
    ctx.sedef_trace_enable(True)
    v = ctx.sedef_filter_autotune(query, g.offsets, rec, srt, off, g.offsets, p)
    names = ctx.sedef_trace_report(reset=True)
    assert 0 <= v < ctx.sedef_filter_variant()[1]
    assert any(x.endswith("k_qpost") for x in names) and not any(x.endswith("k_pos_bits") for x in names)
    recs = oracle.sketch(g.seq, g.offsets, d)
    runs, _ = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert_rows_equal(run_rows(runs), oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=16),
                      "runs")
    assert any(x.endswith("k_pos_bits") for x in ctx.sedef_trace_report(reset=True))
    with pytest.raises(binding.SedefError) as e:  # no target sequence for the third one
        ctx.sedef_filter_autotune(query, [0, 60_000, 120_000, g.length], rec, srt, off, g.offsets,
                                  binding.params(self_mode=2))
    assert e.value.status == -1
    ctx.close()


def test_each_shape_is_timed_once():
    """The shapes with the warp tier are one and the same: timed once, reported as shape 0."""
    torch = need_gpu()
    ctx = binding.Context(0)
    g = synth.small_case(32, lengths=(90_000,), n_sd=4)
    p = binding.params()
    rec = ctx.sedef_sketch(*ctx.sedef_pack(torch.from_numpy(g.seq).to("cuda:0")), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    count = ctx.sedef_filter_variant()[1]
    ctx.sedef_trace_enable(True)
    v = ctx.sedef_filter_autotune(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert v == 0 or count // 2 <= v < count
    timed = [n for k, (n, _) in ctx.sedef_trace_report(reset=True).items() if k.endswith("k_filter_tune")]
    # three times each: the warp tier and four after it, tier 1 and 2 and the four
    assert timed == [3 * (5 + count // 2 * 6)]
    ctx.close()
