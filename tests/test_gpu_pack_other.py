"""Pack of 16-byte stretches with bytes other than ACGTacgt among them, in any number and place."""
import numpy as np
import pytest

import oracle
from paper_1807_00205_gb300 import binding
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [0.02, 0.5, 1.0])
@pytest.mark.parametrize("n", [15, 16, 17, 4096, 100_003])
def test_any_bytes(n, share):
    torch = need_gpu()
    ctx = binding.Context(0)
    rng = np.random.default_rng(n)
    seq = np.frombuffer(b"ACGTacgt", dtype=np.uint8)[rng.integers(0, 8, n)].copy()
    for other in (rng.integers(0, 256, n).astype(np.uint8), np.full(n, ord("N"), np.uint8),
                  np.full(n, ord("n"), np.uint8)):
        s = np.where(rng.random(n) < share, other, seq)
        for got, want in zip(ctx.sedef_pack(torch.from_numpy(s).to("cuda:0")), oracle.pack(s)):
            assert np.array_equal(got.cpu().numpy().view(np.uint32)[:len(want)], want)
    ctx.close()
