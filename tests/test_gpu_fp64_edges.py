"""The all-FP64 multi-CTA class against the oracle where its integer comparisons
could differ: softened and unsoftened centres, a particle at the centre, a box
wrapped, bands of 0 to a half, radii over many decades."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.parity import compare, fp64_rtol
from tests.test_gpu_bins import _nfw, _population

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band", [0.0, 1e-3, 0.3, 0.5])
@pytest.mark.parametrize("soft", [0.0, 0.5])
@pytest.mark.parametrize("box", [0.0, 5e5])
def test_fp64_edges(box, soft, band):
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(23)
    centres = np.array([[0.3, 499999.7, 250000.1], [1e5, 2e5, 3e5]]) if box else np.zeros((3, 3))
    blocks = []
    for k, c in enumerate(centres):
        p, v, r = _nfw(rng, 4500)
        if k == 2:                      # radii from 1e-12 kpc on
            p[:600] *= 10.0 ** rng.uniform(-12.0, 0.0, 600)[:, None]
        if k == 1:
            p[0] = 0.0
        p = p + c
        blocks.append((np.mod(p, box) if box else p, v, r))
    pop = _population(blocks, synth.COORD_F64)
    pop.box = box
    pop.centre = centres
    prm = ahf.params_for(pop, precision=ahf.PREC_FP64)
    prm.r_soft = soft
    prm.band = band
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_ONCHIP_MAX, 0)
    out, prm, ctx, _ = run_gpu(pop, params=prm, ctx=ctx)
    tol = fp64_rtol(pop)
    compare(pop, prm, out["res"], out["bound_idx"], out["phi"], out["removed_iter"], phi_rtol=tol, vir_rtol=tol,
            exact_order=True)
