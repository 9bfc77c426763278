"""Check periods of a few attempts, and solves in calls of a few.

Which kernels a problem's attempts take depends on its check period and not on
how its calls are cut: a single attempt by itself runs stepped where that is
faster, with the bits of the resident launch, and problems whose periods are
too short for resident ones take the two step kernels throughout.
"""
import numpy as np
import pytest

import lpgen
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "T", "Sigma", "ax", "xbar", "ybar")
CHECK = 3  # kernels of a check
CASES = {  # shortest check period that takes the resident plan
    "one_cta": (lambda: lpgen.tiny_random(3), 2),
    "words": (lambda: lpgen.batch_member(9, 701, 1_753), 1),
    "barriers": (lambda: lpgen.row_length_mix(2), 1),
    "both_far": (lambda: lpgen.powerlaw(2, 66_667, 166_667, 1_000_000), 4),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


def _run(lp, stops, **options):
    with lpop.Problem(lp, alpha=1e-4, phi=3, **options) as p:
        for k in stops:
            p.solve(0.0, k)
        return p.get_state(), p.kernel_times()[2]


def _same(a, b):
    assert all(np.array_equal(a[k], b[k]) for k in KEYS)
    assert a["eta"] == b["eta"] and a["k"] == b["k"] and a["attempts"] == b["attempts"]


@pytest.mark.parametrize("case", sorted(CASES))
def test_periods_below_the_shortest_take_the_step_kernels(case):
    make, shortest = CASES[case]
    lp = make()
    for every in sorted({1, shortest, max(shortest - 1, 1)}):
        got, launches = _run(lp, [12], check_every=every)
        step, n = _run(lp, [12], check_every=every, kernel_timing=1)  # timing selects the step kernels
        periods = 12 // every
        assert n == 2 * 12 + CHECK * (1 + periods)
        if every < shortest:
            _same(got, step)
            assert launches == n
        elif every > 1:
            assert launches == periods + CHECK * (1 + periods)


@pytest.mark.parametrize("case", sorted(CASES))
def test_single_attempts_have_the_bits_of_a_period(case):
    make, _ = CASES[case]
    lp = make()
    whole, _ = _run(lp, [40])
    _same(_run(lp, range(1, 41))[0], whole)
    _same(_run(lp, [1, 3, 4, 20, 21, 40])[0], whole)
