"""sedef_chain in a self mode whose index holds other records than the query: the index says what the
target is, as many records and the same sequences or not."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import assert_rows_equal, chain_rows, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("other", ["own", "one strand", "two hashes", "half the hashes", "fewer"])
def test_chain_takes_the_target_from_its_index(mode, other):
    torch = need_gpu()
    ctx = binding.Context(0)
    g = synth.small_case(41, lengths=(120_000, 60_000), n_sd=10, sd_lo=1500, sd_hi=6000, id_lo=0.93)
    d = oracle.params(self_mode=mode)
    p = binding.params_from_dict(d)
    recs = oracle.sketch(g.seq, g.offsets, d)
    runs = oracle.filter_runs(recs, g.offsets, recs, g.offsets, d, threads=8)
    keep = runs[runs[:, oracle.RUN_COLS.index("keep")] == 1]
    own = oracle.chain(runs, recs, g.offsets, recs, g.offsets, d)
    seed = {c: int(x) for c, x in zip(oracle.RUN_COLS, keep[len(keep) // 2])}
    inside = np.flatnonzero((recs[:, 1] >= seed["j_a"]) & (recs[:, 1] <= seed["j_b"] + d["n"] - d["k"]))
    for x, y in zip(inside, inside[1:]):  # the first of the seed's target records that changes a chain
        target = recs.copy()
        if other == "one strand":
            target[x, 2] ^= 1
        elif other == "two hashes":
            target[[x, y], 0] = target[[y, x], 0]
        elif other == "half the hashes":
            target[::2, 0] = np.roll(target[::2, 0], 1)
        elif other == "fewer":
            target = np.delete(target, np.arange(0, len(target), 7), axis=0)
        want = oracle.chain(runs, recs, g.offsets, target, g.offsets, d)
        if other == "own" or not np.array_equal(want, own):
            break
    assert len(want) > 0 and np.array_equal(want, own) == (other == "own")

    def records(rows):
        r = (rows[:, 0].astype(np.uint64) << np.uint64(33)) | (rows[:, 1].astype(np.uint64) << np.uint64(1)) \
            | rows[:, 2].astype(np.uint64)
        return torch.from_numpy(r.view(np.int64)).to("cuda:0")

    v = np.zeros(len(runs), dtype=binding.RUN_DTYPE)
    for c in oracle.RUN_COLS:
        v[c] = runs[:, oracle.RUN_COLS.index(c)]
    srt, off = ctx.sedef_index(records(target), p)
    chains, _ = ctx.sedef_chain(torch.from_numpy(v.view(np.uint8)).to("cuda:0"), len(v), records(recs), g.offsets,
                                srt, off, g.offsets, p)
    assert_rows_equal(chain_rows(chains), want, "chains")
    ctx.close()
