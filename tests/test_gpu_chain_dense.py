"""Chains of seeds whose windows hold about as many records as one warp keeps, and more."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding
from tests.gpu_helpers import assert_rows_equal, cand_rows_global, chain_rows, need_gpu, run_rows
from tests.test_gpu_edges import tandem_genome

pytestmark = pytest.mark.gpu


# records a window on average, of 230 (joined) and 256 (searched): 739, 296, 246, 211
@pytest.mark.parametrize("w", [1, 4, 5, 6])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_dense_windows(mode, w):
    torch = need_gpu()
    ctx = binding.Context(0)
    d = oracle.params(self_mode=mode, w=w)
    d["step"] = 400
    g = tandem_genome(8)
    recs = oracle.sketch(g.seq, g.offsets, d)
    runs = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=16)
    want = oracle.chain(runs, recs, g.offsets, recs, g.offsets, d)
    assert len(want) > 0
    p = binding.params_from_dict(d)
    seq = torch.from_numpy(g.seq).to("cuda:0")
    rec = ctx.sedef_sketch(*ctx.sedef_pack(seq), g.offsets, p, cap=g.length)
    srt, off = ctx.sedef_index(rec, p)
    got, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert_rows_equal(run_rows(got), runs, "runs")
    ctx.sedef_trace_enable(True)
    chains, _ = ctx.sedef_chain(got, n, rec, g.offsets, srt, off, g.offsets, p)
    tried = any(x.endswith("k_chain_seeds") for x in ctx.sedef_trace_report(reset=True))
    ctx.sedef_trace_enable(False)
    assert_rows_equal(chain_rows(chains), want, "chains")
    assert tried == (w == 6 or (w == 5 and mode == 0))
    if mode:
        out = ctx.selfsearch_graph(seq, g.offsets, p).outputs()
        assert_rows_equal(chain_rows(out["chains"]), want, "captured chains")
        cands, _ = ctx.sedef_selfsearch(seq, g.offsets, p)
        assert_rows_equal(cand_rows_global(cands, g.offsets), oracle.merge(want, d), "candidates")
    ctx.close()
