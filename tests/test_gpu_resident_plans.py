"""Which form of plan a problem's attempts take, by the launches they make, and
the forms in which matrix copies are read from global memory.

* FP64 with both copies there: 40 attempts against the oracle and the step kernels
  (which kernel timing selects) within 1e-10, the bar of the free-running tests.
* FP32 with one copy and with both: single attempts from a state of the step
  kernels against theirs within 1e-5, the bar of the mixed-precision tests.
"""
import numpy as np
import pytest

import lpgen
import oracle
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild
from tests.test_gpu_resident import CASES, _close, _options

pytestmark = pytest.mark.gpu

CHECK = 3  # kernels of a check


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


@pytest.mark.parametrize("precision", [lpop.LP_PREC_FP64, lpop.LP_PREC_MIXED])
@pytest.mark.parametrize("case", sorted(CASES))
def test_a_period_is_one_launch(case, precision):
    make, o = CASES[case]
    with lpop.Problem(make(), precision=precision, **_options(o)) as p:
        p.solve(0.0, 128)
        assert p.kernel_times()[2] == 3 * CHECK + 2
        p.solve(0.0, 150)
        assert p.kernel_times()[2] == 4 * CHECK + 3


def test_both_copies_far():
    lp = lpgen.powerlaw(2, 66_667, 166_667, 1_000_000)
    o = dict(alpha=1e-6, phi=20)
    ref = {}

    def trace(P, S):
        if S.attempts == 40:
            ref.update(x=S.x.copy(), y=S.y.copy(), T=S.T.copy(), Sigma=S.Sigma.copy(), ax=S.ax.copy())

    oracle.solve(lp, oracle.Options(**o), tol=0.0, iter_limit=40, trace=trace)
    got = {}
    for timing in (0, 1):
        with lpop.Problem(lp, kernel_timing=timing, **o) as p:
            p.solve(0.0, 40)
            assert p.kernel_times()[2] == 2 * CHECK + (80 if timing else 1)
            got[timing] = p.get_state()
    for key in ref:
        assert _close(got[0][key], ref[key]), f"{key} against the oracle"
    for key in ("x", "y", "T", "Sigma", "ax", "xbar", "ybar"):
        assert _close(got[0][key], got[1][key]), f"{key} against the step kernels"


@pytest.mark.parametrize("size", [(86_666, 216_666, 1_300_000), (100_000, 250_000, 1_500_000), (160_000, 400_000, 1_040_000), (50_000, 125_000, 800_000)])
def test_fp32_attempts_match_the_step_kernels(size):
    lp = lpgen.powerlaw(2, *size)
    o = dict(alpha=1e-4, phi=5, precision=lpop.LP_PREC_MIXED)
    with lpop.Problem(lp, kernel_timing=1, **o) as step, lpop.Problem(lp, **o) as p:
        for k in (1, 4, 7, 20, 63):
            step.solve(0.0, k - 1)
            p.set_state(step.get_state())
            n0 = p.kernel_times()[2]
            p.solve(0.0, k + 1)  # two attempts: a resident launch (one alone may run stepped)
            assert p.kernel_times()[2] == n0 + 1 + CHECK
            step.solve(0.0, k + 1)
            a, b = p.get_state(), step.get_state()
            for key in ("x", "y", "T", "Sigma", "ax", "xbar", "ybar"):
                assert _close(a[key], b[key], 1e-5), (k, key)
            assert a["k"] == b["k"] and a["restarts"] == b["restarts"]
