"""The filter's global path over few and over many windows: how many warps share a window's dense
groups depends on the number of windows."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import assert_rows_equal, need_gpu, run_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    c = binding.Context(0)
    yield c
    c.close()


def to_dev(a):
    return need_gpu().from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def copies(length, seed=3):
    """Pairs and a crowded family, inverted ones among them."""
    rng = np.random.default_rng(seed)
    s = synth.random_bases(rng, length, 0.45)
    unit = synth.random_bases(rng, 900, 0.45)
    for k in range(24):
        at = int(rng.integers(0, length - 1_000))
        c = synth.mutate(rng, unit, 0.97)[:900]
        s[at:at + len(c)] = synth.reverse_complement(c) if k % 3 == 2 else c
    return synth.genome_from_parts([s])


# w = 1: a window has up to 389 records, more than any tier before the global path takes.  Parts of
# a window with 9,728 warps (152 SMs): 32, 32, 16, 8, 2 and 1.
@pytest.mark.parametrize("windows", [1, 150, 160, 600, 3000, 4870])
@pytest.mark.parametrize("mode", [0, 1])
def test_windows_of_many_records(ctx, windows, mode):
    g = copies(60_000)
    step = max(1, (g.length - 400) // (windows - 1)) if windows > 1 else g.length
    d = oracle.params(self_mode=mode, w=1, n=400)
    d["step"] = step
    recs = oracle.sketch(g.seq, g.offsets, d)
    want = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=16)
    p = binding.params_from_dict(d)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p, cap=g.length)
    srt, off = ctx.sedef_index(rec, p)
    runs, _ = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert_rows_equal(run_rows(runs), want, "runs")
    st = ctx.sedef_filter_stats()
    assert st["overflow_windows"] == st["windows"] >= windows


def test_groups_of_many_windows_are_cheap(ctx):
    """The search for dense groups reads the sorted hits once or twice; their sort writes them five
    to seven times."""
    s = np.empty(6_000_000, dtype=np.uint8)
    synth.random_bases_chunked(np.random.default_rng(1), s, 0.45)
    p = binding.params(self_mode=0, w=1)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(s)), [0, len(s)], p, cap=len(s))
    srt, off = ctx.sedef_index(rec, p)
    ctx.sedef_trace_enable(True)
    for _ in range(2):
        ctx.sedef_trace_report(reset=True)
        ctx.sedef_filter(rec, [0, len(s)], rec, srt, off, [0, len(s)], p)
        ms = {k.split(":")[1]: v[1] for k, v in ctx.sedef_trace_report(reset=True).items() if k.startswith("filter")}
    ctx.sedef_trace_enable(False)
    assert ms["k_slow_groups"] < 0.5 * ms["k_rs_pass"], ms


@pytest.mark.parametrize("w", [1, 16])
def test_threshold_of_zero(ctx, w):
    """tau so small that m(s) = 0: a dense group is one hit, and none before the first is read."""
    g = copies(30_000)
    p = binding.params(self_mode=0, w=w, n=400, k=14, query_step=300, delta_m=2.0)
    m = np.ones(400, dtype=np.int32)
    assert ctx.lib.sedef_threshold_table(binding.ctypes.byref(p), m.ctypes.data, 399, None) == 0 and not m.any()
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p, cap=g.length)
    srt, off = ctx.sedef_index(rec, p)
    for v in (0, 12):
        ctx.sedef_filter_variant(v)
        runs, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
        rows = binding.struct_view(runs, binding.RUN_DTYPE)
        assert n == len(rows) and (w == 16 or n > 0)
        assert (rows["j_a"] <= rows["j_b"]).all() and (rows["j_b"].astype(np.int64) + 400 <= g.length).all()
    ctx.sedef_filter_variant(0)
