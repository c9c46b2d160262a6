"""Ensembles whose instances sort at different intervals (what the autotuner picks):
their steps come in many patterns of parities and sorts, and once the recurring
ones are recorded, steps must only replay, whether from the ensemble's graphs or from the
instances' own; the instances still give what they give alone."""
import pytest

from paper_2606_05893_gb300 import workloads as W
from tests.gpu_compare import compare_integer_moments
from tests.test_gpu_ensemble import same_particles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2606_05893_gb300 as p
    p.load_library()
    return p


def instances(intervals):
    wls = [W.config_tiny(seed=40 + i, n_preload=300) for i in range(len(intervals))]
    for w, k in zip(wls, intervals):
        w.sort_interval = k
    return wls


# one interval; two (12 patterns); four (48); more patterns than a handle keeps, for
# few instances and for so many that it keeps eight
@pytest.mark.parametrize("intervals", [(10, 10), (5, 10), (2, 3), (20, 40), (5, 10, 20, 40), (5, 7, 11, 13), (5, 10) * 33],
                         ids=lambda v: f"{len(v)}x{'-'.join(map(str, dict.fromkeys(v)))}")
def test_recording_ends(pkg, intervals):
    sim = pkg.Simulation(instances(intervals), precision=pkg.PIC_MIXED)
    sim.step(400)
    before = pkg.pic_record_count()
    assert before > 0
    sim.step(200)
    assert pkg.pic_record_count() == before
    sim.close()


def test_uneven_intervals_match_separate_handles(pkg):
    wls = instances((2, 3, 5))
    both = pkg.Simulation(wls, cg_rtol=1e-13, cg_maxit=5000)
    alone = [pkg.Simulation(w, cg_rtol=1e-13, cg_maxit=5000) for w in wls]
    for n in (1, 2, 9, 6):  # patterns stepped singly, recorded and replayed, in runs that begin with each
        for s in [both] + alone:
            s.step(n)
        for i, w in enumerate(wls):
            compare_integer_moments(both.moments(i), alone[i].moments())
            same_particles(both, i, alone[i], 0, w.L)
    for s in [both] + alone:
        s.close()
