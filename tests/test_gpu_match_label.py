"""Labelling the second catalogue's ids (ahf_match_catalogs): lists around a
thread's ids in flight, a CTA's round and the round of a halo's CTAs, against the
oracle."""
import numpy as np
import pytest

from oracle import ahf_oracle as O
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

SIZES = [0, 1, 3, 255, 256, 257, 1023, 1024, 1025, 4095, 4096, 4097, 16_383, 16_384, 16_385, 40_000]


@pytest.mark.parametrize("small", [0, 700, 12_000])
def test_lists_of_every_size(small):
    # with `small` lists of 3 more, a halo gets 16 CTAs, 13 of them and one
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(small)
    sizes = SIZES + [3] * small
    ids = rng.permutation(sum(sizes) + 100)
    cut = np.concatenate([[0], np.cumsum(sizes)])
    lists_b = [ids[a:b] for a, b in zip(cut[:-1], cut[1:])]
    lists_a = [np.concatenate([lists_b[k], ids[-50:]]) for k in range(len(SIZES))] + [np.concatenate([x[:2] for x in lists_b[:1000]])]

    def pack(lists):
        cnt = np.array([len(x) for x in lists], dtype=np.int64)
        off = np.concatenate([[0], np.cumsum(cnt)[:-1]]).astype(np.int64)
        return [torch.from_numpy(x).cuda() for x in (np.concatenate(lists).astype(np.int64), off, cnt)]
    ctx = ahf.Context(0)
    best, shared, xi = ctx.match_catalogs(len(ids), *pack(lists_a), *pack(lists_b))
    torch.cuda.synchronize()
    ctx.sync()
    rb, rs, rx = O.match_catalogs(lists_a, lists_b)
    np.testing.assert_array_equal(best.cpu().numpy(), rb)
    np.testing.assert_array_equal(shared.cpu().numpy(), rs)
    np.testing.assert_array_equal(xi.cpu().numpy(), rx)
