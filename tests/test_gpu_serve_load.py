"""Serving under load with the default configuration: requests whose work the
budget spreads over several launches, or leaves whole for the next one, beside
whole requests that hold every SM for a millisecond.  Every residue equals the
same matrix's alone."""
import numpy as np
import pytest

from paper_2407_20205_gb300 import inputs

pytestmark = pytest.mark.gpu

# Gray indices per second of the headline workload, which the offered load is a
# share of; the mean request of n = 12..40 has 2^41 / 29 of them.
CAPACITY = 9.6e14
MEAN_WORK = 2.0 ** 41 / 29


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def mix(pf3):
    from paper_2407_20205_gb300 import serve
    trace = serve.make_trace(inputs.SEED_SERVE + 2, 2500, 12, 40)
    return trace, [pf3.perm_f3(A) for (n, kind, A, parts) in trace]


@pytest.mark.parametrize("rho", [0.7, 0.9, 4.0])
def test_mix_under_load_equals_alone(pf3, mix, rho):
    """Arrivals at a share of the capacity (4.0: far beyond it, so that the
    queue, the slots and every launch's budget are full)."""
    from paper_2407_20205_gb300 import serve
    trace, alone = mix
    for turn in range(4):
        arrivals = inputs.poisson_arrivals(inputs.SEED_SERVE + 3 + turn, len(trace), rho * CAPACITY / MEAN_WORK)
        res = serve.replay(trace, arrivals)[0]
        wrong = [(k, trace[k][0], trace[k][1], res[k], alone[k]) for k in range(len(trace)) if res[k] != alone[k]]
        assert not wrong, wrong[:10]


def test_requests_admitted_by_one_launch_and_run_by_the_next(pf3):
    """Launches with room for one or two requests' work, slots that are used
    again at once, and whole requests in between."""
    mats = [inputs.uniform_matrix(6100, n, k) for k in range(40) for n in (14, 18, 24, 26, 33, 36, 20, 28)]
    mats += [inputs.uniform_matrix(6101, 38), inputs.uniform_matrix(6102, 40)]
    want = [pf3.perm_f3(A) for A in mats]
    for cfg in ({"launch_budget": 1 << 24, "max_jobs": 24}, {"launch_items": 5}, {"max_admit": 3, "launch_budget": 1 << 26}):
        with pf3.ServeContext(**cfg) as ctx:
            for turn in range(3):
                order = np.random.default_rng(turn).permutation(len(mats))
                tickets = [ctx.submit(mats[k]) for k in order]
                assert [ctx.wait(t) for t in tickets] == [want[k] for k in order], (cfg, turn)
