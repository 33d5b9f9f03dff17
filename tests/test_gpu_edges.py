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


def sketch_rows(ctx, g, d):
    p = binding.params_from_dict(d)
    torch = need_gpu()
    packed, mask, nbits = ctx.sedef_pack(to_dev(g.seq))
    rec = ctx.sedef_sketch(packed, mask, nbits, g.offsets, p)
    static = torch.zeros(g.length + 1, dtype=torch.int64, device="cuda:0")
    n = binding.sedef_sketch_noalloc(packed, mask, nbits, g.offsets, p, static,
                                     torch.cuda.current_stream())
    assert n == rec.numel() and torch.equal(static[:n], rec)  # count and write = one pass
    return rec_rows(rec)


# around a lane's 16 positions, whole lanes, the 32-bit keys' limit (112) and the widest
@pytest.mark.parametrize("w", [1, 2, 3, 7, 8, 9, 15, 16, 17, 31, 33, 50, 63, 64, 97, 111, 112, 113,
                               128, 200, 255, 256])
@pytest.mark.parametrize("k", [2, 8, 12, 13, 15])
def test_sketch_window_lengths(ctx, k, w):
    rng = np.random.default_rng(w * 16 + k)
    lengths = [k + w - 2, k + w - 1, k + w, 5, 0, 1, 700, 481, 3841, 9000]
    parts = [synth.random_bases(rng, n) for n in lengths]
    parts[-1][2000:2600] = ord("A")  # equal and palindromic k-mers
    parts[-1][3000:3400] = np.frombuffer(b"ACGT" * 100, dtype=np.uint8)
    g = synth.genome_from_parts(parts)
    s = g.seq
    low = rng.random(len(s)) < 0.4
    s[low] |= 32
    s[rng.integers(0, len(s), 12)] = ord("N")
    for least in (0, 1, 4):
        d = oracle.params(k=k, w=w, min_unmasked=least)
        assert_rows_equal(sketch_rows(ctx, g, d), oracle.sketch(g.seq, g.offsets, d),
                          f"k {k} w {w} min_unmasked {least}")


@pytest.mark.parametrize("n", [479, 480, 481, 3839, 3840, 3841, 15 * 16 * 8 * 40 + 7])
def test_sketch_tile_ends(ctx, n):
    """Window counts around a warp's and a CTA's tile, sequences that end inside one."""
    rng = np.random.default_rng(n)
    for cut in (0, 1, 16, n // 2):
        parts = [synth.random_bases(rng, cut), synth.random_bases(rng, n - cut)]
        g = synth.genome_from_parts(parts)
        d = oracle.params()
        assert_rows_equal(sketch_rows(ctx, g, d), oracle.sketch(g.seq, g.offsets, d), f"{n} {cut}")


def test_pack_every_byte(ctx):
    """Every byte value in every place of a thread's 16, alone among bases."""
    seq = np.frombuffer(b"ACGTacgt" * 2, dtype=np.uint8)
    rows = np.tile(seq, (256 * 16, 1))
    for b in range(256):
        for x in range(16):
            rows[b * 16 + x, x] = b
    flat = np.ascontiguousarray(rows.ravel())
    for got, want in zip(ctx.sedef_pack(to_dev(flat)), oracle.pack(flat)):
        assert np.array_equal(got.cpu().numpy().view(np.uint32)[:len(want)], want)


@pytest.mark.parametrize("pd", [
    dict(k=4, w=3, n=60, step=20, gap_max=60, diag_max=6), dict(k=7, w=5, n=200, step=100),
    dict(k=10, w=4), dict(), dict(self_mode=2), dict(w=40), dict(delta_m=0.02, delta_g=0.02)])
@pytest.mark.parametrize("max_len", [2000, 30_000])
def test_extend_batches(ctx, pd, max_len):
    """Regions that grow over many minimizers at once, end at a sequence's end, at the cap, where
    the two would overlap, or where the estimate falls; small hash tables."""
    from tests.test_gpu_extend import gpu_extend
    rng = np.random.default_rng(3)
    a = synth.random_bases(rng, 45_000, 0.45)
    a[20_000:29_000] = synth.mutate(rng, a[4_000:14_000], 0.97)[:9_000]
    a[36_000:45_000] = synth.reverse_complement(synth.mutate(rng, a[5_000:15_000], 0.9)[:9_000])
    a[30_000:33_000] = np.tile(a[30_000:30_900], 4)[:3_000]   # mates that meet
    b = synth.random_bases(rng, 12_000, 0.45)
    b[:6_000] = synth.mutate(rng, a[8_000:15_000], 0.93)[:6_000]
    g = synth.genome_from_parts([a, b])
    d = oracle.params(**pd)
    recs = oracle.sketch(g.seq, g.offsets, d)
    runs = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=8)
    keep = np.flatnonzero(runs[:, oracle.RUN_COLS.index("keep")] == 1)
    pick = keep[np.unique(np.linspace(0, len(keep) - 1, 40).astype(np.int64))]
    allk = oracle.sketch(g.seq, g.offsets, dict(d, min_unmasked=0))
    want = oracle.extend(runs[pick], allk, g.offsets, allk, g.offsets, d, max_len=max_len, threads=16)
    got, _ = gpu_extend(ctx, g, d, max_len, keep_runs=pick)
    assert len(want) == len(pick) > 0
    assert_rows_equal(got, want, "regions")


def test_chain2_item_counts(ctx):
    """Regions with no seed, one, and around 32 and 256 of them; long ones with many chains."""
    from tests.test_gpu_chain2 import sd_rows
    rng = np.random.default_rng(12)
    s = synth.random_bases(rng, 120_000)
    s[60_000:100_000] = synth.mutate(rng, s[2_000:44_000], 0.9)[:40_000]
    s[100_500:108_000] = synth.reverse_complement(synth.mutate(rng, s[5_000:13_000], 0.95)[:7_500])
    s[110_000:116_000] = np.tile(s[110_000:110_037], 200)[:6_000]
    g = synth.genome_from_parts([s])
    rows = []
    for n in [0, 5, 11, 12, 40, 90, 200, 300, 400, 700, 1200, 2000, 2600, 3300, 5000, 20_000, 40_000]:
        rows.append((2_000, 2_000 + n, 60_000, 60_000 + n, 0))
        m = min(n, 7_400)
        rows.append((5_000, 5_000 + m, 108_000 - m, 108_000, 1))
        m = min(n, 1_200)
        rows.append((110_000, 110_000 + m, 112_000, 112_000 + m, 0))
    v = np.zeros(len(rows), dtype=binding.REGION_DTYPE)
    for c, x in zip(("qa", "qb", "ta", "tb", "o"), np.array(rows).T):
        v[c] = x
    ext = np.stack([v[c].astype(np.int64) for c in oracle.EXTEND_COLS], axis=1)
    want = oracle.chain2(g.seq, ext, threads=16)
    packed, _, nbits = ctx.sedef_pack(to_dev(g.seq))
    out, _ = ctx.sedef_chain2(packed, nbits, g.length, to_dev(v.view(np.uint8)), len(v),
                              binding.params())
    assert len(want) > 15
    assert_rows_equal(sd_rows(out), want, "SDs")


def crowded_genome(seed=9):
    """Windows with few hits, around 2,048 of them (the warp tier's most), with a counter past
    255 and with more than 256 collected: families of copies of one element, of many sizes."""
    rng = np.random.default_rng(seed)
    seq = synth.random_bases(rng, 260_000, 0.45)
    at = 2_000
    for copies in (2, 5, 12, 20, 24, 28, 40, 70):
        unit = synth.random_bases(rng, 800, 0.45)
        for _ in range(copies):
            pc = synth.mutate(rng, unit, float(rng.uniform(0.9, 1.0)))
            if rng.random() < 0.4:
                pc = synth.reverse_complement(pc)
            seq[at:at + len(pc)] = pc
            at += len(pc) + int(rng.integers(0, 700))
    seq[at:at + 4_000] = np.tile(synth.random_bases(rng, 25, 0.5), 160)
    return synth.genome_from_parts([seq[:150_000], seq[150_000:]])


@pytest.mark.parametrize("pd", [dict(), dict(w=11), dict(w=40), dict(k=9, w=20), dict(k=14),
                                dict(delta_m=0.5, delta_g=0.5, w=60, step=700),
                                dict(delta_m=0.9, delta_g=0.2, w=60, step=700), dict(max_occ=30)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_filter_crowded_windows(ctx, pd, mode):
    """Every self mode (target starts before the window too, when overlap > n), eager and captured."""
    d = oracle.params(self_mode=mode, **pd)
    g = crowded_genome()
    recs = oracle.sketch(g.seq, g.offsets, d)
    want = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=16)
    assert len(want) > 100
    p = binding.params_from_dict(d)
    seq = to_dev(g.seq)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(seq), g.offsets, p)
    srt, off = ctx.sedef_index(rec, p)
    runs, _ = ctx.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    assert_rows_equal(run_rows(runs), want, "runs")
    if mode and not pd.get("delta_m"):
        out = ctx.selfsearch_graph(seq, g.offsets, p).outputs()
        assert_rows_equal(run_rows(out["runs"]), want, "captured runs")


def test_filter_under_scratch_caps(ctx):
    """With too little scratch for the record posting ranges the tiers look postings up themselves,
    with less the refine runs fewer warps and then its large kernel alone: the same runs down to
    the cap where the call is refused."""
    g = crowded_genome()
    p = binding.params()
    c = binding.Context(0)
    rec = c.sedef_sketch(*c.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, off = c.sedef_index(rec, p)
    want, n = c.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p)
    want, refused = want.cpu(), 0
    caps = np.geomspace(64 << 20, 32 << 10, 100).astype(np.int64)
    c.sedef_trace_enable(True)
    names = set()
    for nbytes in caps:
        c.sedef_set_scratch_limit(0)
        c.sedef_set_scratch_limit(int(nbytes))
        try:
            runs, m = c.sedef_filter(rec, g.offsets, rec, srt, off, g.offsets, p, cap=n + 1)
        except binding.SedefError as e:
            assert e.status == -2
            refused += 1
            continue
        names |= set(c.sedef_trace_report(reset=True))
        assert m == n and bool((runs.cpu() == want).all())
    assert 0 < refused < len(caps)
    assert any(x.endswith("k_refine_all") for x in names), names
    c.close()


@pytest.mark.parametrize("mode", [1, 2])
def test_graph_record_overflow(ctx, mode):
    """A captured pass whose record capacity is far too small: every kernel keeps to the records
    that were written, the totals come back, and a graph rebuilt with them gives the eager pass."""
    g = synth.small_case(17, lengths=(90_000, 40_000), n_sd=6, sd_lo=2000, sd_hi=8000, mask_frac=0.2)
    p = binding.params(self_mode=mode)
    d = to_dev(g.seq)
    eager = ctx.selfsearch(d, g.offsets, p)
    caps = {k: 1 << 20 for k in binding.CAP_NAMES}
    caps["records"] = 3
    gr = binding.Graph(ctx, d, g.offsets, p, caps)
    gr.launch()
    with pytest.raises(binding.SedefError) as e:
        gr.wait()
    assert e.value.status == binding.SEDEF_ERR_CAPACITY
    assert gr.need["records"] == eager["rec"].numel()
    gr.close()
    out = ctx.selfsearch_graph(d, g.offsets, p, caps={k: 1 for k in binding.CAP_NAMES}).outputs()
    assert np.array_equal(run_rows(out["runs"]), run_rows(eager["runs"]))


@pytest.mark.parametrize("n", [1, 31, 257, 4095, 4096, 4097, 8192, 40_961, 1_300_003])
@pytest.mark.parametrize("k", [2, 4, 8, 11, 13])
def test_index_sort_sizes(ctx, n, k):
    """The sort below, at and past one CTA's keys, over one to four passes, with digits that are
    spread, skewed and all alike; equal hashes stay by position."""
    torch = need_gpu()
    rng = np.random.default_rng(n + k)
    top = 4 ** k
    for h in (rng.integers(0, top, n), (rng.random(n) ** 8 * top).astype(np.int64),
              np.full(n, top - 1), np.sort(rng.integers(0, top, n))[::-1]):
        rec = (h.astype(np.uint64) << np.uint64(33)) | (np.arange(n, dtype=np.uint64) * np.uint64(3) << np.uint64(1)) \
            | rng.integers(0, 2, n).astype(np.uint64)
        srt, off = ctx.sedef_index(to_dev(rec.view(np.int64)), binding.params(k=k))
        want = rec[np.argsort(h, kind="stable")]
        assert np.array_equal(srt.cpu().numpy().view(np.uint64), want)
        cnt = np.concatenate([[0], np.cumsum(np.bincount(h, minlength=top))])
        assert bool((off.cpu().to(torch.int64) == torch.from_numpy(cnt)).all())


@pytest.mark.parametrize("pd", [dict(), dict(w=5), dict(w=2, n=400, step=200), dict(w=40), dict(k=9, w=8),
                                dict(gap_max=60, diag_max=5), dict(max_occ=20), dict(min_unmasked=3)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("which", ["tandem", "crowded"])
def test_chain_anchor_counts(ctx, which, pd, mode):
    """Seeds with a few anchors, around 32 and past the 256 that one warp keeps, with more than 256
    query records, joined (self modes) and searched, on both strands."""
    from tests.gpu_helpers import chain_rows
    d = oracle.params(self_mode=mode, **pd)
    g = tandem_genome(6) if which == "tandem" else crowded_genome(10)
    recs = oracle.sketch(g.seq, g.offsets, d)
    runs = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=16)
    runs = runs[::max(1, len(runs) // 400)]
    want = oracle.chain(runs, recs, g.offsets, recs, g.offsets, d)
    p = binding.params_from_dict(d)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p)
    srt, tab = ctx.sedef_index(rec, p)
    v = np.zeros(len(runs), dtype=binding.RUN_DTYPE)
    for c in oracle.RUN_COLS:
        v[c] = runs[:, oracle.RUN_COLS.index(c)]
    chains, n = ctx.sedef_chain(to_dev(v.view(np.uint8)), len(v), rec, g.offsets, srt, tab, g.offsets, p)
    assert_rows_equal(chain_rows(chains), want, "chains")


def test_posting_ranges_parted(ctx):
    """A batch with more records than the posting ranges are parted from (16 M): the candidates of
    its genomes searched alone (fewer records each)."""
    from paper_1807_00205_gb300 import batch
    rng = np.random.default_rng(77)
    parts = []
    for n in (41_000_003, 17_000_001):
        s = np.empty(n, dtype=np.uint8)
        synth.random_bases_chunked(rng, s, 0.45)
        for _ in range(60):
            a, b = rng.integers(0, n - 9_000, 2)
            c = synth.mutate(rng, s[a:a + 8_000], float(rng.uniform(0.85, 1.0)))
            s[b:b + len(c)] = synth.reverse_complement(c)[:n - b] if rng.random() < 0.5 else c[:n - b]
        parts.append(s)
    g = synth.genome_from_parts(parts)
    p = binding.params(w=5, self_mode=2)
    both = to_dev(g.seq)
    rec = ctx.sedef_sketch(*ctx.sedef_pack(both), g.offsets, p)
    assert rec.numel() > 16 << 20
    cands, n = ctx.sedef_selfsearch(both, g.offsets, p)
    rows = batch.split_candidates(binding.struct_view(cands, binding.CAND_DTYPE), 2)
    assert n > 100
    for k, s in enumerate(parts):
        alone, m = ctx.sedef_selfsearch(to_dev(s), [0, len(s)], binding.params(w=5))
        assert np.array_equal(binding.struct_view(alone, binding.CAND_DTYPE), rows[k]), k


@pytest.mark.parametrize("copies", [16, 24, 35, 70, 105, 150, 640])
@pytest.mark.parametrize("gap", [0, 1200])
def test_filter_many_copies(ctx, copies, gap):
    """Windows whose collected hits come around what each shape of the CTA tier, the tier after it
    and the global path hold, in one dense group on each strand and in one per copy; with the
    shared memory of every tier, of the ones beside a serving kernel, and of the smallest ones."""
    rng = np.random.default_rng(copies + gap)
    unit = synth.random_bases(rng, 1_500, 0.45)
    parts = []
    for k in range(copies):
        pc = synth.mutate(rng, unit, 0.98)
        parts += [synth.reverse_complement(pc) if k % 5 == 4 else pc,
                  synth.random_bases(rng, gap + int(rng.integers(0, 40)), 0.45)]
    target = synth.genome_from_parts([np.concatenate(parts), synth.random_bases(rng, 5_000, 0.45)])
    query = synth.genome_from_parts([np.concatenate([synth.random_bases(rng, 600, 0.45), unit,
                                                     synth.random_bases(rng, 500, 0.45)])])
    d = oracle.params(self_mode=0)
    qrec, trec = (oracle.sketch(g.seq, g.offsets, d) for g in (query, target))
    want = oracle.filter_runs(qrec, query.offsets, trec, target.offsets, d, threads=16)
    assert len(want) >= 4
    p = binding.params_from_dict(d)
    dq, dt = (ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p).clone() for g in (query, target))
    srt, off = ctx.sedef_index(dt, p)
    c = binding.Context(0)
    for nbytes in (-1, 180_000, 100 * 1024):
        c.sedef_set_tier_smem_limit(nbytes)
        runs, _ = c.sedef_filter(dq, query.offsets, dt, srt, off, target.offsets, p)
        assert_rows_equal(run_rows(runs), want, f"runs with {nbytes} bytes of shared memory")
    c.close()


def test_refine_crowded_rank(ctx):
    """More than 255 hashes of a target window between two neighbours of W_Q (here all below the
    first): past the batched kernel's counters, so its runs go to the large one."""
    d = oracle.params(self_mode=0, w=5, n=1000)  # windows of 989 starts
    rng = np.random.default_rng(5)
    unit = np.frombuffer(b"GATTCTG", dtype=np.uint8)
    q = np.full(1_600, ord("N"), dtype=np.uint8)
    q[700:900] = np.tile(unit, 29)[:200]
    t = np.concatenate([synth.random_bases(rng, 100, 0.45), np.tile(unit, 7)[:45],
                        synth.random_bases(rng, 1_500, 0.45)])
    query, target = synth.genome_from_parts([q]), synth.genome_from_parts([t])
    qrec, trec = (oracle.sketch(g.seq, g.offsets, d) for g in (query, target))
    wq, inside = np.unique(qrec[:, 0]), trec[trec[:, 1] < 989][:, 0]
    assert np.bincount(np.searchsorted(wq, np.setdiff1d(inside, wq)))[0] > 255
    want = oracle.filter_runs(qrec, query.offsets, trec, target.offsets, d)
    assert len(want) == 3
    p = binding.params_from_dict(d)
    dq, dt = (ctx.sedef_sketch(*ctx.sedef_pack(to_dev(g.seq)), g.offsets, p).clone() for g in (query, target))
    srt, off = ctx.sedef_index(dt, p)
    runs, _ = ctx.sedef_filter(dq, query.offsets, dt, srt, off, target.offsets, p)
    assert_rows_equal(run_rows(runs), want, "runs")
    assert ctx.sedef_filter_stats()["big_refine"] == len(want)
