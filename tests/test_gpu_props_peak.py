"""The rotation curve's peak (ahf_halo_properties): in units whose squares leave
the range of a float, against the oracle; and where thousands of particles tie
to rounding, the same bytes from every call."""
import dataclasses

import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu
from tests.test_gpu_bins import _population
from tests.test_gpu_props import _check_props, _run

pytestmark = pytest.mark.gpu


def _scaled(pop, length, mass, velocity):
    """The population and the method's parameters in other units."""
    from paper_0904_3662_gb300 import ahf
    base = ahf.Params()
    new = dataclasses.replace(
        pop, **{k: getattr(pop, k) * length for k in "xyz"}, **{k: getattr(pop, k) * velocity for k in ("vx", "vy", "vz")},
        m=None if pop.m is None else (pop.m * mass).astype(pop.m.dtype), m0=pop.m0 * mass, centre=pop.centre * length,
        radius=pop.radius * length, r200=pop.r200 * length)
    return new, dict(G=base.G * length * velocity ** 2 / mass, H=base.H * velocity / length,
                     delta_rho=base.delta_rho * mass / length ** 3)


@pytest.mark.parametrize("masses", [False, True])
def test_peak_in_si_units(masses):
    # metres, kilograms, m/s: r^2 ~ 1e42 and M ~ 1e41 lie beyond a float
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    pop = synth.halo_batch(seed=85, n_halos=16, n_lo=100, n_hi=10_000, coord_type=synth.COORD_F64, with_masses=masses)
    si, kw = _scaled(pop, 3.0857e19, 1.989e30, 1e3)
    _, prm, _, host = _run(si, precision=ahf.PREC_FP64, **kw)
    assert _check_props(si, prm, host, 1e-11) >= 14


@pytest.mark.parametrize("length,mass", [(1.0, 1e-26), (1e-10, 1e-33)])
def test_peak_with_small_masses(length, mass):
    # M^2 / r^2, or M^2 alone, below a normal float
    pop = synth.halo_batch(seed=86, n_halos=16, n_lo=100, n_hi=10_000, with_masses=True)
    small, kw = _scaled(pop, length, mass, 1.0)
    _, prm, _, host = _run(small, **kw)
    assert _check_props(small, prm, host, 1e-5) >= 14


@pytest.mark.parametrize("masses", [False, True])
def test_peak_of_a_flat_curve_is_repeatable(masses):
    # M(<= r_i) / r_i the same to rounding for every particle: the first of the
    # largest, whatever order the threads come in
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    n = 2048
    pos = np.zeros((n, 3))
    pos[:, 0] = 0.01 * np.arange(1, n + 1)
    pop = _population([(pos, np.zeros((n, 3)), 100.0)] * 32, synth.COORD_F64)
    if masses:
        pop.m = np.full(pop.n_particles, pop.m0)
    ctx, prm, out, host = _run(pop, precision=ahf.PREC_FP64, H=0.0)
    assert np.all(host["props"][:, 0] == n)
    parts, hal = ahf.particles_from_population(pop), ahf.halos_from_population(pop)
    for _ in range(20):
        props = ctx.halo_properties(parts, hal, prm, out)
        assert props.cpu().numpy().tobytes() == host["props"].tobytes()
    assert np.all(host["props"] == host["props"][0])       # (32 equal haloes)
