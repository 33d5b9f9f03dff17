"""Scratch caps: a cap that suffices keeps sufficing when it is raised, and buffers that a call can
do without (posting ranges, refine events) are not what it fails for."""
import numpy as np
import pytest

from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


def to_dev(a):
    return need_gpu().from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def genome(mode):
    return synth.small_case(5, lengths=(600_000, 300_000) if mode == 1 else (300_000,) * 3, n_sd=40,
                            sd_lo=2000, sd_hi=9000, mask_frac=0.25)


def accepted(ctx, caps, call):
    """Which caps `call` passes under; any other outcome than success and OOM is an error."""
    ok = np.zeros(len(caps), dtype=bool)
    for k, cap in enumerate(caps):
        ctx.sedef_set_scratch_limit(0)
        ctx.sedef_set_scratch_limit(int(cap))
        try:
            call()
            ok[k] = True
        except binding.SedefError as e:
            assert e.status == -2, e  # SEDEF_ERR_OOM
    return ok


# windows every few bases, so that the ranges pay
@pytest.mark.parametrize("pd", [dict(query_step=20), dict(k=13, query_step=20), dict(w=3, n=300, query_step=10),
                                dict(self_mode=2, query_step=40), dict(self_mode=2, k=14, query_step=40)])
def test_filter_caps(pd):
    ctx = binding.Context(0)
    g = genome(pd.get("self_mode", 1))
    p = binding.params(**pd)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    want, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    want = want.cpu()
    # the records' ranges alone are 8 bytes each, what a window and a run need less than 64 and 128;
    # the caps reach below that
    windows = ctx.sedef_filter_stats()["windows"]
    with_per_window = 64 * windows + 128 * n
    caps = np.geomspace(16 * windows, 128 << 20, 120).astype(np.int64)
    ctx.sedef_trace_enable(True)
    with_ranges = []

    def call():
        ctx.sedef_trace_report(reset=True)
        runs, m = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p, cap=n + 1)
        assert m == n and bool((runs.cpu() == want).all())
        with_ranges.append(any(x.endswith("k_pos_bits") for x in ctx.sedef_trace_report(reset=True)))

    ok = accepted(ctx, caps, call)
    first = int(np.argmax(ok))
    assert ok[first:].all(), caps[first:][~ok[first:]]
    assert caps[first] < with_per_window + 8 * rec.numel()
    assert not with_ranges[0] and with_ranges[-1]
    ctx.close()


def test_stage_after_stage_caps():
    """One context through the whole search: what the filter could do without is there for the
    calls after it."""
    ctx = binding.Context(0)
    g = genome(1)
    p = binding.params(query_step=20)
    d = to_dev(g.seq)
    want = binding.struct_view(ctx.sedef_selfsearch(d, g.offsets, p)[0], binding.CAND_DTYPE)
    out = ctx.selfsearch(d, g.offsets, p)

    def call():
        runs, n = ctx.sedef_filter(out["rec"], g.offsets, out["rec"], out["sorted"], out["off"], g.offsets, p,
                                   cap=out["nruns"] + 1)
        chains, m = ctx.sedef_chain(runs, n, out["rec"], g.offsets, out["sorted"], out["off"], g.offsets, p)
        cands, _ = ctx.sedef_merge(chains, m, g.offsets, g.offsets, p)
        assert np.array_equal(binding.struct_view(cands, binding.CAND_DTYPE), want)

    caps = np.geomspace(100 << 10, 64 << 20, 120).astype(np.int64)
    ok = accepted(ctx, caps, call)
    first = int(np.argmax(ok))
    assert 0 < first and ok[first:].all(), caps[first:][~ok[first:]]

    def whole():
        assert np.array_equal(binding.struct_view(ctx.sedef_selfsearch(d, g.offsets, p)[0],
                                                  binding.CAND_DTYPE), want)

    caps = np.linspace(64 << 20, 84 << 20, 160).astype(np.int64)  # the offset table alone: 64 MB and 4 bytes
    ok = accepted(ctx, caps, whole)
    first = int(np.argmax(ok))
    assert 0 < first and ok[first:].all(), caps[first:][~ok[first:]]
    ctx.close()


@pytest.mark.parametrize("mode", [1, 2])
def test_graph_caps(mode):
    """A captured pass is recorded without the ranges and events where the cap has no room for them."""
    ctx = binding.Context(0)
    g = genome(mode)
    p = binding.params(self_mode=mode, query_step=100)
    d = to_dev(g.seq)
    want = ctx.selfsearch(d, g.offsets, p)
    rows = binding.struct_view(want["cands"], binding.CAND_DTYPE)
    need = dict(records=want["rec"].numel(), slow_hits=1000, runs=want["nruns"],
                anchors=40 * want["nruns"] + 1000, chains=want["nchains"], cands=want["ncands"])
    nodes = []

    def call():
        gr = binding.Graph(ctx, d, g.offsets, p, need)
        gr.launch()
        gr.wait()
        assert np.array_equal(binding.struct_view(gr.outputs()["cands"], binding.CAND_DTYPE), rows)
        nodes.append(gr.nodes)
        gr.close()

    caps = np.geomspace(1 << 20, 32 << 20, 250).astype(np.int64)
    ok = accepted(ctx, caps, call)
    first = int(np.argmax(ok))
    assert 0 < first and ok[first:].all(), caps[first:][~ok[first:]]
    assert nodes[0] < nodes[-1]
    ctx.close()


def test_server_caps():
    """A served request under the caps of the server's context."""
    ctx = binding.Context(0)
    g = synth.small_case(8, lengths=(400_000,), n_sd=20, sd_lo=2000, sd_hi=9000)
    p = binding.params(self_mode=0)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    query = g.seq[50_000:230_000]
    rows = []

    def call():
        srv = binding.DeviceServer(ctx, rec, srt, off, g.offsets, p, slots=1, slot_bases=200_000)
        try:
            slot = srv.submit(query)
            assert srv.poll(5.0) == slot
            rows.append(srv.finish(slot))
        finally:
            srv.close()

    caps = np.geomspace(64 << 10, 16 << 20, 60).astype(np.int64)
    ok = accepted(ctx, caps, call)
    first = int(np.argmax(ok))
    assert 0 < first and ok[first:].all(), caps[first:][~ok[first:]]
    assert len(rows[0]) > 0 and all(np.array_equal(r, rows[-1]) for r in rows)
    ctx.close()


def test_parted_ranges_caps():
    """More records than the ranges are parted from (16 M), with room for the parts and not for the
    sort's own scratch: the ranges go straight to their records, so the hits looked at are as many
    as without a cap (without ranges they would be about twice as many)."""
    torch = need_gpu()
    ctx = binding.Context(0)
    rng = np.random.default_rng(2)
    s = np.empty(17_400_000, dtype=np.uint8)
    synth.random_bases_chunked(rng, s, 0.5)
    for at in range(0, 200_000, 10_000):
        s[9_000_000 + at:9_004_000 + at] = s[at:at + 4_000]
    g = synth.genome_from_parts([s])
    p = binding.params(w=1, n=100, query_step=60)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(s)), g.offsets, p, cap=len(s))
    assert rec.numel() > 16 << 20
    srt, off = ctx.sedef_index(rec, p)
    ctx.sedef_trace_enable(True)

    def run(cap):
        ctx.sedef_set_scratch_limit(0)
        ctx.sedef_set_scratch_limit(int(cap))
        ctx.sedef_trace_report(reset=True)
        runs, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p, cap=1 << 20)
        placed = any(x.endswith("k_qpost_place") for x in ctx.sedef_trace_report(reset=True))
        return runs.cpu(), ctx.sedef_filter_stats()["hits"], placed

    want, hits, placed = run(4 << 30)
    assert placed and len(want) > 0
    lo, hi = 256 << 20, 4 << 30  # the smallest cap under which the parts are placed
    while hi - lo > 64 << 10:
        mid = (lo + hi) // 2
        if run(mid)[2]:
            hi = mid
        else:
            lo = mid
    # the sort's scratch is half a byte a record
    for cap in (lo, lo - rec.numel() // 4, lo - rec.numel() // 2 + (64 << 10), lo - rec.numel()):
        runs, n, placed = run(cap)
        assert not placed and n == hits, cap
        assert torch.equal(runs, want), cap
    ctx.close()


def test_merge_caps():
    """Scratch of the merge: 56 bytes a chain and its sort's 12.5, 52 a candidate."""
    ctx = binding.Context(0)
    g = synth.small_case(6, lengths=(700_000, 500_000), n_sd=60, sd_lo=2000, sd_hi=9000, mask_frac=0.25)
    p = binding.params(self_mode=0, query_step=100)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    runs, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    chains, m = ctx.sedef_chain(runs, n, rec, g.offsets, srt, off, g.offsets, p)
    cands, nc = ctx.sedef_merge(chains, m, g.offsets, g.offsets, p)
    assert m > 4096
    small = 24 << 10  # offsets, the sorts' heads, each array rounded up to 256 bytes

    def merge():
        got, k = ctx.sedef_merge(chains, m, g.offsets, g.offsets, p)
        assert k == nc and np.array_equal(got.cpu(), cands.cpu())

    assert accepted(ctx, [68.5 * m + 52 * nc + (12.5 * nc if nc > 4096 else 0) + small], merge).all()
    ctx.close()


@pytest.mark.parametrize("pd", [dict(self_mode=0, query_step=100), dict(w=1, n=500, query_step=500)])
def test_chain_caps(pd):
    """Scratch of the chain: 52 bytes a run, 16 an anchor of the seeds past what one warp holds (in a
    self-search 256 query records: a window of 500 bases has 489 of them at w = 1)."""
    ctx = binding.Context(0)
    g = synth.small_case(6, lengths=(700_000, 500_000), n_sd=60, sd_lo=2000, sd_hi=9000)
    p = binding.params(**pd)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p, cap=g.length)
    srt, off = ctx.sedef_index(rec, p)
    runs, n = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    # many of the same seeds, so that the bytes a run count
    runs = runs.reshape(n, -1).repeat(128, 1).reshape(-1)
    n *= 128
    args = (runs, n, rec, g.offsets, srt, off, g.offsets, p)
    ctx.sedef_trace_enable(True)
    chains, m = ctx.sedef_chain(*args)
    big = any(x.endswith("k_anchor_fill") for x in ctx.sedef_trace_report(reset=True))
    assert big == (p.w == 1)
    anchors = ctx.sedef_filter_stats()["anchors"] if big else 0
    keep = int(binding.struct_view(runs, binding.RUN_DTYPE)["keep"].sum())
    assert 4 * keep > 64 << 10  # so that four bytes a kept run more would show
    small = 24 << 10  # offsets, table, each array rounded up to 256 bytes, the scan's sums

    def chain():
        got, k = ctx.sedef_chain(*args)
        assert k == m and np.array_equal(got.cpu(), chains.cpu())

    assert accepted(ctx, [52 * n + 16 * anchors + small], chain).all()
    ctx.close()
