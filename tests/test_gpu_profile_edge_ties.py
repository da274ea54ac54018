"""Profile rows where a shell of equal radii lies on a bin edge: the count at the
edge is found by halving, not member by member."""
import math
import time

import numpy as np
import pytest

from oracle import ahf_oracle as O
from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu
from tests.parity import oracle_params
from tests.test_gpu_bins import _population

pytestmark = pytest.mark.gpu

N_BINS, F_MIN = 2, 0.0625                                  # one inner edge, a quarter of r_out


def _halo(n, n_shell, at):
    """n cold particles spread well inside and n_shell of them at the radius `at`."""
    rng = np.random.default_rng(n)
    d = rng.standard_normal((n, 3))
    d *= (rng.uniform(1e-3, 0.5, n) * at / np.linalg.norm(d, axis=1))[:, None]
    u = np.array([3.0, 4.0, 5.0]) / math.sqrt(50.0) * at
    d[:n_shell] = np.where(rng.uniform(size=(n_shell, 3)) < 0.5, -1.0, 1.0) * u
    return _population([(d, np.zeros((n, 3)), 2.0 * at)], synth.COORD_F32_REL)


@pytest.mark.parametrize("n,n_shell", [(400, 350), (3000, 2500), (100_000, 60_000), (700_000, 600_000)])
def test_profile_with_a_shell_on_a_bin_edge(n, n_shell):
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    # all of it inside r_vir = (M / (4 pi / 3 delta_rho))^(1/3): the edge is known
    base = ahf.Params()
    r_vir = (n * synth.PARTICLE_MASS / (4.0 * math.pi / 3.0 * base.delta_rho)) ** (1.0 / 3.0)
    edge = r_vir * math.sqrt(F_MIN)
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_PROMOTE, 0)
    took = {}
    for where, at in (("on", edge), ("off", edge * 0.98)):
        pop = _halo(n, n_shell, at)
        prm = ahf.params_for(pop, H=0.0)
        parts, hal = ahf.particles_from_population(pop), ahf.halos_from_population(pop)
        best = math.inf
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            out = ctx.unbind_profile_batch(parts, hal, prm, n_bins=N_BINS, r_min_frac=F_MIN)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        ctx.sync()
        took[where] = best
        res, prof = ahf.results_to_numpy(out["res"]), out["prof"].cpu().numpy()[0]
        assert res[0]["n_bound"] == n and res[0]["r_vir"] == pytest.approx(r_vir, rel=1e-12)
        assert prof[:, 0].sum() == n - np.sum(_radii(pop) <= r_vir * F_MIN)
        if where == "off":
            o = O.unbind_population(pop, oracle_params(prm), n_bins=N_BINS, r_min_frac=F_MIN)[0]["profile"]
            np.testing.assert_array_equal(prof[:, 0], o[:, 0])
            np.testing.assert_allclose(prof[:, 1:], o[:, 1:], rtol=1e-5)
        else:
            # the shell falls on one side of the edge, whole
            assert prof[1, 0] in (0.0, float(n_shell))
    assert took["on"] < 2.0 * took["off"], took


def _radii(pop):
    return np.sqrt(pop.x.astype(np.float64) ** 2 + pop.y.astype(np.float64) ** 2 + pop.z.astype(np.float64) ** 2)
