"""Recorded steps: after the first step (which deposits from scratch), steps that
neither sort nor time their phases are recorded once per buffer parity and then
replayed as one graph launch each. The replays must give what direct steps give
(against the FP64 oracle at the parity tolerance), including across sort steps,
source changes (the carries move between host and device) and both precisions."""
import numpy as np
import pytest

import oracle as O
from paper_2606_05893_gb300 import workloads as W
from tests.gpu_compare import compare_integer_moments, compare_particles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2606_05893_gb300 as p
    p.load_library()
    return p


def test_replayed_steps_match_oracle(pkg):
    wl = W.config_small(seed=21, n_preload=4000)
    wl.sort_interval = 5
    sim = pkg.Simulation(wl, cg_rtol=1e-13, cg_maxit=5000)
    ref = O.Oracle(wl, cg_rtol=1e-13)
    sim.step(2)
    ref.step(2)
    l0, k0 = pkg.pic_launch_count(), pkg.pic_kernel_count()
    sim.step(2)  # steps 2, 3: recorded (two buffer parities)
    sim.step(2)  # steps 4, 5: a replay and a sort step
    sim.step(2)  # steps 6, 7: replays
    launches = pkg.pic_launch_count() - l0
    kernels = pkg.pic_kernel_count() - k0
    ref.step(6)
    mg, mo = sim.moments(), ref.moments()
    compare_integer_moments(mg, mo)
    for sp in range(3):
        compare_particles(sim, ref, wl, sp, 1e-9, 1e-9)
    assert np.abs(sim.phi() - ref.phi()).max() <= 1e-9 * np.abs(ref.phi()).max()
    # 5 recorded or replayed steps cost one launch each, for some tens of
    # kernels each; the sort step is enqueued directly
    assert kernels - launches >= 5 * 20, (launches, kernels)
    sim.close()


def test_source_change_between_replays(pkg):
    wl = W.config_small(seed=22, n_preload=3000)
    sim = pkg.Simulation(wl, cg_rtol=1e-13, cg_maxit=5000)
    ref = O.Oracle(wl, cg_rtol=1e-13)
    sim.step(4)
    ref.step(4)
    # a stronger electron source from now on (both sides keep their carries)
    src = wl.sources[0]
    pkg.pic_inject(sim.h, 0, 0, src.cx, src.cy, src.radius, src.flux_m2s * 37.0, src.T_K)
    ref.set_source(0, src.flux_m2s * 37.0, src.T_K)
    sim.step(4)
    ref.step(4)
    compare_integer_moments(sim.moments(), ref.moments())
    for sp in range(3):
        compare_particles(sim, ref, wl, sp, 1e-9, 1e-9)
    sim.close()


def test_mixed_replays_keep_counts(pkg):
    wl = W.config_small(seed=23, n_preload=3000)
    sim = pkg.Simulation(wl, precision=pkg.PIC_MIXED)
    direct = pkg.Simulation(wl, precision=pkg.PIC_MIXED)
    pkg.pic_set_profiling(direct.h, True)  # timed steps are always enqueued directly
    sim.step(6)
    direct.step(6)
    a, b = sim.moments(), direct.moments()
    for k in ("count", "injected", "abs_cathode", "abs_anode", "next_pid"):
        assert a[k] == b[k], k
    sim.close()
    direct.close()


def test_autotuner_times_every_candidate_from_the_same_state():
    """The autotuner restores every instance before each candidate and once at the
    end: the run continues from where it was (exact checkpoint round trip), and a
    second call finds every bucket cached and runs no step."""
    import paper_2606_05893_gb300 as pkg
    from paper_2606_05893_gb300 import autotune
    from paper_2606_05893_gb300 import workloads as W
    wls = [W.config_tiny(seed=11), W.config_tiny(seed=12, nx=8, ny=8, nz=24)]
    sim = pkg.Simulation(wls, precision=pkg.PIC_MIXED)
    sim.step(3)
    before = [sim.moments(i) for i in range(2)]
    parts = [[sim.particles(sp, i) for sp in range(3)] for i in range(2)]
    cache = {}
    chosen, measured = autotune.tune(sim, intervals=(5, 20), shapes=(4, 8), window=6, cache=cache)
    assert len(measured) == 4 and all(c in measured for c in chosen)
    for i in range(2):
        m = sim.moments(i)
        assert m["step"] == before[i]["step"] and m["count"] == before[i]["count"]
        assert m["pushed"] == before[i]["pushed"]
        for sp in range(3):
            x, v, p = sim.particles(sp, i)
            x0, v0, p0 = parts[i][sp]
            o, o0 = np.argsort(p), np.argsort(p0)
            assert np.array_equal(p[o], p0[o0]) and np.array_equal(x[o], x0[o0]) and np.array_equal(v[o], v0[o0])
    chosen2, measured2 = autotune.tune(sim, intervals=(5, 20), shapes=(4, 8), window=6, cache=cache)
    assert measured2 == {} and chosen2 == chosen
    assert sim.moments(0)["step"] == before[0]["step"]
    sim.step(2)
    sim.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_recorded_sort_of_an_overfull_cell(pkg, precision):
    """Sort steps are recorded too; a cell of more than 4096 particles sends its species to the radix
    sort, which sits in a conditional node there. Steps with and without recording end alike."""
    from tests._cases import bare
    wl = bare(nx=4, ny=4, nz=8, weight=1e-6, capacity=1 << 14, phi_a=1.0)
    wl.sort_interval = 2
    rng = np.random.default_rng(3)

    def cloud(n):
        dense = (np.array([1, 2, 3]) + 0.05 + 0.9 * rng.random((n, 3))) * wl.h
        return np.concatenate([dense, rng.random((500, 3)) * np.array(wl.L)]), rng.standard_normal((n + 500, 3)) * 10.0

    wl.preload = [cloud(5000), cloud(20), cloud(4500)]
    a = pkg.Simulation(wl, precision=precision, cg_rtol=1e-12)
    b = pkg.Simulation(wl, precision=precision, cg_rtol=1e-12)
    pkg.pic_set_profiling(b.h, True)  # timed steps are always enqueued directly
    a.step(9)
    b.step(9)
    for sp in range(3):
        xa, va, pa = a.particles(sp)
        xb, vb, pb = b.particles(sp)
        oa, ob = np.argsort(pa), np.argsort(pb)
        assert np.array_equal(pa[oa], pb[ob]) and len(np.unique(pa)) == pa.size
        # deposits sum in another order: FP64 rounding, or the mixed store's parity bounds per step
        tol_x, tol_v = (1e-10 * max(wl.L), 1e-10) if precision == 0 else (9 * 1e-5 * wl.h, 9 * 1e-5)
        assert np.abs(xa[oa] - xb[ob]).max() <= tol_x
        assert np.abs(va[oa] - vb[ob]).max() <= tol_v * np.abs(va).max()
    a.sort_now()
    x, v, pid = a.particles(0)
    cell = np.minimum((x / wl.h).astype(int), np.array([3, 3, 7]))
    key = (cell[:, 2] * 4 + cell[:, 1]) * 4 + cell[:, 0]
    assert np.all(np.lexsort((pid, key)) == np.arange(pid.size))
    a.close()
    b.close()
