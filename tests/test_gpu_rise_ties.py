"""The edge at the rise of the density profile (AHF_VAR_RISE_EDGE) in thread-block
clusters, where the record's CTA reads the radii that other CTAs hold, with
hundreds of equal radii in single shells: a CTA whose share holds them sorts by
another way than its neighbours."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.parity import compare

pytestmark = pytest.mark.gpu


def _tie(pop, n, shells, ties):
    """`ties` particles of each of the given shells of n moved to the radius of one."""
    rng = np.random.default_rng(n)
    for s in shells:
        at = s * n + np.arange(ties)
        p = np.stack([pop.x[at], pop.y[at], pop.z[at]], axis=1)
        mid = np.abs(p[ties // 2])
        p = np.where(rng.uniform(size=p.shape) < 0.5, -mid, mid).astype(np.float32)
        pop.x[at], pop.y[at], pop.z[at] = p[:, 0], p[:, 1], p[:, 2]
    return pop


@pytest.mark.parametrize("shells", [(5, 9), (9, 13), (6, 8, 10, 11)])
@pytest.mark.parametrize("n,cls", [(800, "cluster2_16k"), (1250, "cluster4_32k"), (2500, "cluster8_64k"),
                                   (5000, "cluster16_128k")])
def test_rise_edge_with_equal_radii_in_clusters(n, cls, shells):
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    pop = _tie(synth.shell_profile_batch(n_shells=(n,)), n, shells, 250)
    out, prm, ctx, _ = run_gpu(pop, params=ahf.params_for(pop, variant=ahf.VAR_RISE_EDGE))
    assert ctx.stats()["phase_halos"][ahf.PHASE_NAMES.index(cls)] == 1
    compare(pop, prm, out["res"], out["bound_idx"], out["phi"], out["removed_iter"])
    assert out["res"][0]["status"] == ahf.HALO_RVIR_BEYOND_EDGE | ahf.HALO_RISE_EDGE
    assert out["res"][0]["k_vir"] == 12 * n - 1
