"""On-chip classes launched as a chain on one stream against the same classes one
after another (AHF_OPT_SERIAL): every class present, single classes, gaps in the
order, more haloes than one class holds at once, a multi-CTA halo beside the
chain, replayed graphs, and calls that follow each other without a
synchronisation.  The sums are exact, so every output byte must agree."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu
from tests.test_gpu_bins import _nfw, _population

pytestmark = pytest.mark.gpu

CLASSES = {
    "all": [300, 900, 3000, 8000, 16_000, 30_000, 60_000, 120_000],
    "one": [900] * 3,
    "gap": [120_000, 16_000, 300, 300],
    "more_than_resident": [700] * 1200 + [9000] * 90 + [200] * 3000,
    "with_grid": [300_000, 120_000, 3000, 300],
}


def _run(ahf, torch, pop, serial, graphs, repeats):
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_PROMOTE, 0)
    ctx.set_option(ahf.OPT_SERIAL, int(serial))
    ctx.set_option(ahf.OPT_GRAPHS, int(graphs))
    parts = ahf.particles_from_population(pop)
    hal = ahf.halos_from_population(pop)
    prm = ahf.params_for(pop)
    outs = []
    for _ in range(repeats):                # zeroed: slots past a halo's bound count are not written
        out = ctx.alloc_outputs(len(hal), int(hal["count"].sum()), True, True, prm.precision)
        outs.append({k: v.zero_() for k, v in out.items() if v is not None})
    prof = [torch.zeros((len(hal), 16, 4), dtype=torch.float64, device="cuda") for _ in range(repeats)]
    outs = [ctx.unbind_profile_batch(parts, hal, prm, n_bins=16, r_min_frac=0.01, out=o, prof=q)
            for o, q in zip(outs, prof)]
    torch.cuda.synchronize()
    ctx.sync()
    return [{k: o[k].cpu().numpy().tobytes() for k in ("res", "phi", "removed_iter", "bound_idx", "prof")} for o in outs]


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("shape", list(CLASSES))
def test_chain_equals_serial(shape, graphs):
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(77)
    pop = _population([_nfw(rng, n) for n in CLASSES[shape]], synth.COORD_F32_REL, False)
    ref = _run(ahf, torch, pop, True, False, 1)[0]
    for out in _run(ahf, torch, pop, False, graphs, 3):
        for k in ref:
            assert out[k] == ref[k], k
