"""A sort tile whose wait for the tiles before it runs out counts their keys itself.

With no polls every tile that does not find its predecessors' counts at once takes that way, so the
calls that sort must give what they give with the default, in records, runs and candidates.
"""
import ctypes

import numpy as np
import pytest

from paper_1807_00205_gb300 import binding, synth
from tests.gpu_helpers import need_gpu, run_rows

pytestmark = pytest.mark.gpu


def set_polls(ctx, polls):
    f = ctx.lib.sedef_debug_sort_polls
    f.argtypes = [ctypes.c_void_p, ctypes.c_int32]
    assert f(ctx.handle, polls) == 0


@pytest.fixture()
def ctx():
    need_gpu()
    c = binding.Context(0)
    yield c
    c.close()


def to_dev(a):
    return need_gpu().from_numpy(np.ascontiguousarray(a)).to("cuda:0")


# two tiles, a ragged last one, more tiles than the look-back reads at once, than run side by side
@pytest.mark.parametrize("n", [4097, 8193, 40_960, 200_001, 3_000_017])
@pytest.mark.parametrize("polls", [0, 1])
def test_index_counts_for_itself(ctx, n, polls):
    rng = np.random.default_rng(n)
    k = 11
    top = 4 ** k
    for h in (rng.integers(0, top, n), (rng.random(n) ** 8 * top).astype(np.int64)):
        rec = (h.astype(np.uint64) << np.uint64(33)) | (np.arange(n, dtype=np.uint64) << np.uint64(1))
        set_polls(ctx, polls)
        srt, off = ctx.sedef_index(to_dev(rec.view(np.int64)), binding.params(k=k))
        assert np.array_equal(srt.cpu().numpy().view(np.uint64), rec[np.argsort(h, kind="stable")])
        assert int(off[top]) == n


@pytest.mark.parametrize("mode", [1, 2])
def test_pass_counts_for_itself(ctx, mode):
    """Keys with payloads (runs, candidates), eager and captured."""
    g = synth.small_case(23, lengths=(900_000, 400_000), n_sd=120, sd_lo=2000, sd_hi=9000, mask_frac=0.2)
    p = binding.params(self_mode=mode, query_step=60)
    d = to_dev(g.seq)
    want = ctx.selfsearch(d, g.offsets, p)
    assert len(run_rows(want["runs"])) > 4096
    set_polls(ctx, 0)
    got = ctx.selfsearch(d, g.offsets, p)
    captured = ctx.selfsearch_graph(d, g.offsets, p).outputs()
    for name, dtype in (("runs", binding.RUN_DTYPE), ("chains", binding.CHAIN_DTYPE),
                        ("cands", binding.CAND_DTYPE)):
        rows = binding.struct_view(want[name], dtype)
        assert np.array_equal(binding.struct_view(got[name], dtype), rows), name
        assert np.array_equal(binding.struct_view(captured[name], dtype), rows), name
