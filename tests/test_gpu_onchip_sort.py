"""The on-chip classes' radial sort against the oracle: halo sizes at and next to
each class's capacity with every candidate a member, equal radii by the dozen
(ordered among themselves) and by the hundred (left to the radix sort), a
particle at the centre, all radii equal."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.parity import compare
from tests.test_gpu_bins import _nfw, _population

pytestmark = pytest.mark.gpu

FULL = [1, 2, 31, 33, 511, 512, 513, 1023, 1024, 1025, 4095, 4096, 4097, 8191, 8192, 8193, 16383, 16384, 16385, 32768]
TIED = [300, 1000, 3000, 8000, 16000, 30000]


def _blocks(shapes):
    rng = np.random.default_rng(31)
    blocks = []
    if shapes == "full":
        return [_nfw(rng, n) for n in FULL]
    for n in TIED:
        p, v, r = _nfw(rng, n)
        p[0] = 0.0
        ties = {"dozens": 40, "hundreds": 250, "all": n}[shapes]
        sign = np.where(rng.uniform(size=(ties, 3)) < 0.5, -1.0, 1.0)
        p[n - ties:] = sign * np.array([3.0, 4.0, 5.0]) * (0.1 * r / 5.0)
        blocks.append((p, v, r))
    return blocks


@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("shapes", ["full", "dozens", "hundreds", "all"])
def test_onchip_sort_against_oracle(shapes, masses):
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    pop = _population(_blocks(shapes), synth.COORD_F32_REL, masses)
    out, prm, ctx, _ = run_gpu(pop)
    st = ctx.stats()
    assert st["phase_halos"][ahf.PHASE_NAMES.index("grid_gather_sort")] == 0
    compare(pop, prm, out["res"], out["bound_idx"], out["phi"], out["removed_iter"])
