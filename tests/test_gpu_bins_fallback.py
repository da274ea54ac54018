"""The multi-CTA class where radii are equal by the hundred, against the oracle:
around what a part of a radial bin holds (its bin is then ordered by comparisons),
in a halo of one tile (one bin, a map of its own) and of several; and by the
thousand, more than a bin holds, where the radix sort takes over.  With gas and
member lists, whose arrays the ordering of a bin reads by the places it has found."""
import numpy as np
import pytest

from paper_0904_3662_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu
from tests.parity import compare, fp64_rtol
from tests.test_gpu_bins import _nfw, _population

pytestmark = pytest.mark.gpu

PART = 512                                                 # members of a part ordered by counting
BIN = 3072                                                 # members of a bin


def _shell(rng, n, ties):
    """n particles, the first `ties` of them at one radius, the others well inside."""
    d = rng.standard_normal((n, 3))
    d *= (rng.uniform(5.0, 35.0, n) / np.linalg.norm(d, axis=1))[:, None]
    d[:ties] = np.where(rng.uniform(size=(ties, 3)) < 0.5, -1.0, 1.0) * np.array([30.0, 40.0, 50.0])
    return d, 20.0 * rng.standard_normal((n, 3)), 100.0


def _shuffled(pop, rng):
    """The particle store in another order, and the member list that undoes it."""
    perm = rng.permutation(pop.n_particles).astype(np.int64)
    for k in ("x", "y", "z", "vx", "vy", "vz", "m", "u_th"):
        a = getattr(pop, k)
        if a is not None:
            b = np.empty_like(a)
            b[perm] = a
            setattr(pop, k, b)
    return perm


def _run(pop, mode, member_idx=None):
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    fp64 = mode == "fp64"
    prm = ahf.params_for(pop, precision=ahf.PREC_FP64 if fp64 else ahf.PREC_MIXED)
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_ONCHIP_MAX, 0)                  # every halo to the multi-CTA class
    out, prm, ctx, _ = run_gpu(pop, params=prm, ctx=ctx, member_idx=member_idx)
    tol = fp64_rtol(pop) if fp64 else 1e-5
    compare(pop, prm, out["res"], out["bound_idx"], out["phi"], out["removed_iter"], member_idx=member_idx,
            phi_rtol=tol, vir_rtol=tol, exact_order=fp64)
    # the radix sort reads the keys' range back: two synchronisations more
    # than the reads of the pass chunks (8 passes each)
    return ctx.stats(), ctx.stats()["host_syncs"] - -(-int(out["res"]["n_iter"].max()) // 8) >= 2


def _coord(mode):
    return synth.COORD_F64 if mode == "fp64" else synth.COORD_F32_REL


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("n,ties", [(600, PART), (600, PART + 1), (1024, 1023), (2000, 1025), (2000, 2000),
                                    (5000, PART + 1), (9000, 1500), (9000, BIN + 1)])
def test_equal_radii_around_what_a_part_and_a_bin_hold(n, ties, mode):
    pop = _population([_shell(np.random.default_rng(n + ties), n, ties)], _coord(mode))
    _, radix = _run(pop, mode)
    assert radix == (ties > BIN)


@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("gas,members", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("thousands", [False, True])
def test_equal_radii_with_gas_and_member_lists(thousands, gas, members, mode, masses):
    rng = np.random.default_rng(41)
    blocks = [_nfw(rng, 3000), _shell(rng, 5000, 900), _shell(rng, 700, 650), _nfw(rng, 300)]
    pop = _population(blocks + [_shell(rng, 9000, 4000)] * thousands, _coord(mode), masses)
    if gas:
        pop = synth.with_gas(pop, frac=0.3, u_max=1e3)
    _, radix = _run(pop, mode, _shuffled(pop, rng) if members else None)
    assert radix == thousands


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_abandoned_bins_do_not_count_as_iterations(mode):
    st = {}
    for ties in (PART, BIN + 1):
        pop = _population([_shell(np.random.default_rng(7), 6000, ties)], _coord(mode))
        st[ties], radix = _run(pop, mode)
        assert radix == (ties > BIN)
    # (8 passes to a chunk; each halo needs one chunk)
    assert st[PART]["grid_iterations"] == st[BIN + 1]["grid_iterations"] == 8


def test_radix_sort_after_bins_is_timed_as_sort():
    require_gpu()
    from paper_0904_3662_gb300 import ahf
    pop = _population([_shell(np.random.default_rng(53), 300_000, 100_000)], synth.COORD_F64)
    ctx = ahf.Context(0)
    ctx.set_option(ahf.OPT_TIMING, 1)
    run_gpu(pop, params=ahf.params_for(pop, precision=ahf.PREC_FP64, max_iter=1), ctx=ctx)
    st = ctx.stats()
    sort, iterate = (ahf.PHASE_NAMES.index(k) for k in ("grid_gather_sort", "grid_iterate"))
    assert st["phase_halos"][sort] == st["phase_halos"][iterate] == 1
    # eight radix passes against one pass of the iteration
    assert st["phase_ms"][sort] > 2.0 * st["phase_ms"][iterate]


def test_one_halo_with_equal_radii_leaves_the_others_in_bins():
    # (the radix sort of every halo takes about as long as the whole call in bins)
    torch = require_gpu()
    import time
    from paper_0904_3662_gb300 import ahf
    rng = np.random.default_rng(43)
    blocks = [_nfw(rng, int(n)) for n in rng.integers(300, 3000, 3000)]
    took, outs = [], []
    for ties in (PART, 900):
        pop = _population(blocks[:1500] + [_shell(np.random.default_rng(3), 1200, ties)] + blocks[1500:], synth.COORD_F64)
        prm = ahf.params_for(pop, precision=ahf.PREC_FP64)
        ctx = ahf.Context(0)
        parts, hal = ahf.particles_from_population(pop), ahf.halos_from_population(pop)
        out = ctx.alloc_outputs(pop.n_halos, pop.n_particles, precision=ahf.PREC_FP64)
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            ctx.unbind_batch(parts, hal, prm, out=out)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        took.append(best)
        res = ahf.results_to_numpy(out["res"])
        host = [out[k].cpu().numpy() for k in ("bound_idx", "phi", "removed_iter")]
        tol = fp64_rtol(pop)
        compare(pop, prm, res, *host, halos=[0, 700, 1499, 1500, 1501, 3000], phi_rtol=tol, vir_rtol=tol,
                exact_order=True)
        outs.append((res, host))
    (ra, ha), (rb, hb) = outs
    rest = np.arange(3001) != 1500
    assert ra[rest].tobytes() == rb[rest].tobytes()
    slot = np.repeat(rest, pop.count)
    np.testing.assert_array_equal(ha[2][slot], hb[2][slot])
    assert took[1] < 1.5 * took[0], took


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_most_of_a_large_halo_at_one_radius(mode):
    # (counted one by one on one address, 1.8e6 members took five times the untied call)
    torch = require_gpu()
    import time
    from paper_0904_3662_gb300 import ahf
    fp64 = mode == "fp64"
    n = 2_000_000
    took = []
    for ties in (0, 1_800_000):
        rng = np.random.default_rng(47)
        p, v, r = _shell(rng, n, ties)
        order = rng.permutation(n)
        pop = _population([(p[order], v[order], r)], _coord(mode))
        prm = ahf.params_for(pop, precision=ahf.PREC_FP64 if fp64 else ahf.PREC_MIXED)
        ctx = ahf.Context(0)
        parts, hal = ahf.particles_from_population(pop), ahf.halos_from_population(pop)
        out = ctx.alloc_outputs(1, n, precision=prm.precision)
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            ctx.unbind_batch(parts, hal, prm, out=out)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        took.append(best)
    tol = fp64_rtol(pop) if fp64 else 1e-5
    compare(pop, prm, ahf.results_to_numpy(out["res"]), *[out[k].cpu().numpy() for k in ("bound_idx", "phi", "removed_iter")],
            phi_rtol=tol, vir_rtol=tol, exact_order=fp64)
    assert took[1] < 3.0 * took[0], took
