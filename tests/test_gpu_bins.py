"""The multi-CTA class's radial order by distribution into bins, against the
oracle: halo sizes around a tile, the two bins of a small halo, the change of
cell counts at 8 tiles; ties within a part; and radii the bins cannot hold
(hundreds equal, a thin shell in a void), which go to the radix sort."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.parity import compare, fp64_rtol

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 511, 513, 2047, 2048, 2049, 4095, 4097, 14336, 14337, 16385]


def _population(blocks, coord_type, masses=False):
    count = np.array([len(p) for p, _, _ in blocks], dtype=np.int64)
    offset = np.concatenate([[0], np.cumsum(count)[:-1]]).astype(np.int64)
    pos = np.concatenate([p for p, _, _ in blocks])
    vel = np.concatenate([v for _, v, _ in blocks])
    dt = np.float64 if coord_type == synth.COORD_F64 else np.float32
    m = None
    if masses:
        m = synth.PARTICLE_MASS * np.exp(np.random.default_rng(5).uniform(-1.0, 1.0, len(pos)))
    n = len(blocks)
    return synth.Population(
        name="bins", coord_type=coord_type, **{k: pos[:, a].astype(dt) for a, k in enumerate("xyz")},
        **{k: vel[:, a].astype(dt) for a, k in enumerate(("vx", "vy", "vz"))},
        m=None if m is None else m.astype(dt), m0=synth.PARTICLE_MASS, box=0.0, centre=np.zeros((n, 3)),
        radius=np.array([r for _, _, r in blocks]), offset=offset, count=count, r200=np.zeros(n), conc=np.zeros(n))


def _nfw(rng, n):
    n_cont = n // 8
    p, v, r200 = synth._halo_block(rng, n - n_cont, n_cont, 10.0, synth.PARTICLE_MASS)
    return p, v, 2.0 * r200


def _blocks(shapes):
    rng = np.random.default_rng(11)
    if shapes == "sizes":
        return [_nfw(rng, n) for n in SIZES]
    blocks = []
    # a particle at the centre; 60 and 300 particles at one radius (one part)
    for ties in (60, 300):
        p, v, r = _nfw(rng, 5000)
        p[0] = 0.0
        p[1000:1000 + ties] = np.where(rng.uniform(size=(ties, 3)) < 0.5, -1.0, 1.0) * np.array([30.0, 40.0, 50.0])
        blocks.append((p, v, r))
    if shapes == "overflow":
        # 900 at one radius: more than a part may hold
        p, v, r = _nfw(rng, 5000)
        p[1000:1900] = np.where(rng.uniform(size=(900, 3)) < 0.5, -1.0, 1.0) * np.array([30.0, 40.0, 50.0])
        blocks.append((p, v, r))
        # a thin shell, a little mass far outside and inside it
        d = rng.standard_normal((6000, 3))
        d /= np.linalg.norm(d, axis=1)[:, None]
        s = 100.0 * (1.0 + 1e-5 * rng.uniform(size=6000))
        s[:5] = [1e-3, 1e-2, 1.0, 3e3, 1e4]
        blocks.append((d * s[:, None], 5.0 * rng.standard_normal((6000, 3)), 2e4))
    return blocks


@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("shapes", ["sizes", "ties", "overflow"])
def test_bins_against_oracle(shapes, mode, masses):
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    fp64 = mode == "fp64"
    pop = _population(_blocks(shapes), synth.COORD_F64 if fp64 else synth.COORD_F32_REL, masses)
    prm = ahf.params_for(pop, precision=ahf.PREC_FP64 if fp64 else ahf.PREC_MIXED)
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_ONCHIP_MAX, 0)                  # every halo to the multi-CTA class
    out, prm, ctx, _ = run_gpu(pop, params=prm, ctx=ctx)
    st = ctx.stats()
    assert st["phase_halos"][ahf.PHASE_NAMES.index("grid_gather_sort")] == pop.n_halos
    # the radix sort reads the keys' range back: two synchronisations more
    # than the reads of the pass chunks (8 passes each)
    extra = st["host_syncs"] - -(-int(out["res"]["n_iter"].max()) // 8)
    assert (extra >= 2) == (shapes == "overflow")
    tol = fp64_rtol(pop) if fp64 else 1e-5
    compare(pop, prm, out["res"], out["bound_idx"], out["phi"], out["removed_iter"], phi_rtol=tol, vir_rtol=tol,
            exact_order=fp64)
