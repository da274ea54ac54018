"""Properties, profiles and matching at the edges of their kernels' chunks:
bound sets of a chunk (4,096) and of one CTA round, one less and one more, a
particle at the centre; match lists around a CTA's round with labels that
change at every id."""
import numpy as np
import pytest

from oracle import ahf_oracle as O
from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu
from tests.parity import check_profiles
from tests.test_gpu_props import _check_props, _run

pytestmark = pytest.mark.gpu

SIZES = [255, 256, 257, 1023, 1025, 4095, 4096, 4097, 8193]


def _cold(coord_type, masses):
    """Cold uniform spheres (nothing unbinds without the Hubble flow), one
    particle of each at its centre where the offsets are exact (float32 relative
    coordinates)."""
    rng = np.random.default_rng(21)
    count = np.array(SIZES, dtype=np.int64)
    offset = np.concatenate([[0], np.cumsum(count)[:-1]]).astype(np.int64)
    n = int(count.sum())
    dt = np.float64 if coord_type == synth.COORD_F64 else np.float32
    centre = rng.uniform(0.0, 1e4, (len(count), 3)) if coord_type == synth.COORD_F64 else np.zeros((len(count), 3))
    pos, vel = np.empty((n, 3)), np.empty((n, 3))
    for h, (o, c) in enumerate(zip(offset, count)):
        p, v = synth.sample_uniform_sphere(rng, int(c), 20.0, 1.0)
        if coord_type != synth.COORD_F64:
            p[c // 2] = 0.0
        pos[o:o + c], vel[o:o + c] = p + centre[h], v
    m = synth.PARTICLE_MASS * np.exp(rng.uniform(-1.0, 1.0, n)) if masses else None
    return synth.Population(
        name="cold", coord_type=coord_type, **{k: pos[:, a].astype(dt) for a, k in enumerate("xyz")},
        **{k: vel[:, a].astype(dt) for a, k in enumerate(("vx", "vy", "vz"))}, m=None if m is None else m.astype(dt),
        m0=synth.PARTICLE_MASS, box=0.0, centre=centre, radius=np.full(len(count), 25.0), offset=offset, count=count,
        r200=np.zeros(len(count)), conc=np.zeros(len(count)))


@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("coord", ["f32", "f64"])
def test_properties_and_profile_chunk_edges(coord, masses):
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    pop = _cold(synth.COORD_F64 if coord == "f64" else synth.COORD_F32_REL, masses)
    ctx, prm, out, host = _run(pop, H=0.0)
    assert np.array_equal(host["res"]["n_bound"], pop.count)
    assert _check_props(pop, prm, host, 1e-5) >= len(SIZES) - 2
    prof = ctx.profile_batch(ahf.particles_from_population(pop), ahf.halos_from_population(pop), prm, out["res"],
                             out["bound_idx"], n_bins=48, r_min_frac=0.01)
    torch.cuda.synchronize()
    check_profiles(pop, prm, host["res"], prof.cpu().numpy(), 48, 0.01)


def test_match_labels_change_at_every_id():
    torch = require_gpu()
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(22)
    n_b, per = 300, 40
    ids = rng.permutation(n_b * per + 500)
    lists_b = [ids[k * per:(k + 1) * per] for k in range(n_b)]
    lists_a = [rng.permutation(ids)[:n] for n in (0, 1, 511, 512, 513, 2047, 2048, 2049, 12_000)]

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
