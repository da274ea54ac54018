"""The multi-CTA class's FP32 recentring against the exact fixed-point one of the
on-chip classes: the same haloes through both must give the same bytes.  Centres
that are floats (ties of the rounding), that are not, next to the box's faces
(candidates wrapped), on a face; coordinates off the fixed-point grid, zero,
outside every frame and not finite; a frame without a box."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.test_gpu_bins import _nfw, _population

pytestmark = pytest.mark.gpu

BOX = 5e5
CENTRES = {
    "float": [[262144.0, 131072.5, 300000.25], [4096.0, 4096.0, 4096.0]],
    "double": [[262144.0 / 3.0, 1e5 * np.pi, 4e5 / 7.0], [123.456789, 0.1, 1.0 / 3.0]],
    "faces": [[0.3, 499999.7, 250000.1], [499990.123, 12.3, 0.05], [0.0, 0.0, 5e5]],
}


@pytest.mark.parametrize("box", [BOX, 0.0])
@pytest.mark.parametrize("where", list(CENTRES))
def test_recentring_same_bytes(where, box):
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(19)
    centres = np.array(CENTRES[where])
    blocks = []
    for c in centres:
        p, v, r = _nfw(rng, 5000)
        p = p + c
        if box:
            p = np.mod(p, box)
        p[10] = 0.0
        p[11, 0] = 1e-6                 # off the grid of 2^-41
        p[12, 1] = -1e-20
        p[13, 2] = 1e-42                # subnormal
        p[14, 0] = 3e30
        p[15, 1] = np.inf
        p[16, 2] = np.nan
        p[17] = c                       # at the centre (rounded to float)
        blocks.append((p, v, r))
    pop = _population(blocks, synth.COORD_F32_BOX if box else synth.COORD_F32_REL)
    pop.box = box
    pop.centre = centres
    outs = []
    for onchip in (True, False):
        ctx = ahf.Context(0)
        ctx.set_option(ahf.OPT_PROMOTE, 0)
        if not onchip:
            ctx.set_option(ahf.OPT_ONCHIP_MAX, 0)
        out, _, ctx, _ = run_gpu(pop, ctx=ctx)
        n = ctx.stats()["phase_halos"][ahf.PHASE_NAMES.index("grid_gather_sort")]
        assert n == (0 if onchip else len(blocks))
        outs.append(out)
    a, b = outs
    assert np.all(a["res"]["n_member"] > 4000)
    assert a["res"].tobytes() == b["res"].tobytes()
    assert a["removed_iter"].tobytes() == b["removed_iter"].tobytes()
    for h, (o, nb) in enumerate(zip(pop.offset, a["res"]["n_bound"])):
        assert np.array_equal(a["bound_idx"][o:o + nb], b["bound_idx"][o:o + nb]), h
        assert np.array_equal(a["phi"][o:o + nb], b["phi"][o:o + nb]), h
