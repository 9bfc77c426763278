"""Resident check periods whose waits run out or whose launch is refused.

In the checked build the limits of the waits can be made short, and an arrival
or a word can be awaited that nothing ever sends (lpop_resident_limits): the
kernel gives up after the limit, sets its error status and returns.  A refused
launch is an error code in the place of the call.  Nothing faults or hangs.
"""
import subprocess
import sys

import pytest

from paper_2506_17650_gb300 import build as lpbuild
from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

PRELUDE = r'''
import ctypes, sys
import numpy as np
root, lib, case = sys.argv[1:4]
sys.path.insert(0, root)
import lpgen
import paper_2506_17650_gb300 as lpop
lpop.load_library(lib)
raw = ctypes.CDLL(lib)
lps = {
    "one_cta": lambda: lpgen.tiny_random(3),
    "words": lambda: lpgen.batch_member(9, 701, 1_753),
    "barriers": lambda: lpgen.row_length_mix(2),
    "far": lambda: lpgen.powerlaw(2, 50_000, 125_000, 800_000),
}
KEYS = ("x", "y", "T", "Sigma", "ax", "xbar", "ybar", "GT", "GS")


def limits(p, **k):
    args = [k.get(n, 0) for n in ("start_spins", "spins", "missing_arrivals", "missing_words", "refuse")]
    assert raw.lpop_resident_limits(p.handle, *args) == 0


def error(fn):
    try:
        fn()
    except lpop.LpError as e:
        return e.code
    return None


lp = lps[case.split("/")[0]]()
options = dict(alpha=1e-4, phi=7, precision=case.endswith("/mixed"))
p = lpop.Problem(lp, **options)
'''


def _run(script, case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = lpbuild.build(checked=True)
    subprocess.run([sys.executable, "-c", PRELUDE + script, ROOT, lib, case], check=True, timeout=600)


LOST = r'''
p.solve(0.0, 64)
start = p.get_state()
limits(p, spins=500, missing_words=1)
assert error(lambda: p.solve(0.0, 128)) == lpop.LP_ERR_CUDA
limits(p)
with lpop.Batch([p]) as b:
    for call in (lambda: p.solve(0.0, 192), p.result, p.get_state, p.iterate, lambda: b.round(0.0, 64, 192)):
        assert error(call) == lpop.LP_ERR_CUDA, call
p.set_state(start)
again = p.get_state()
assert all(np.array_equal(again[k], start[k]) for k in KEYS)
p.solve(0.0, 128)
assert p.get_state()["attempts"] == 128
p.reset()
p.solve(0.0, 64)
x, y, st = p.result()
assert st["iterations"] == 64 and np.all(np.isfinite(x)) and np.all(np.isfinite(y))
'''


@pytest.mark.parametrize("case", ["words", "barriers", "far"])
def test_state_lost_in_a_period_is_refused_until_it_is_set_again(case):
    _run(LOST, case)


NOT_STARTED = r'''
p.close()
more = (dict(), dict(mode=lpop.LP_MODE_PLAIN, scheduler=lpop.LP_SCHED_ADAGRAD_NORM, normalize=0, use_graph=0),
        dict(scheduler=lpop.LP_SCHED_CONST, restart=0, check_every=16, phi=1))
for extra in more:
    opts = dict(options, **extra)
    with lpop.Problem(lp, **opts) as p, lpop.Problem(lp, **opts) as q:
        limits(p, **dict(start_spins=500, missing_arrivals=1) if start else dict(refuse=1))
        for stop in (64, 100, 256):
            n0 = [x.kernel_times()[2] for x in (p, q)]
            p.solve(0.0, stop)
            q.solve(0.0, stop)
            a, b = p.get_state(), q.get_state()
            assert all(np.array_equal(a[k], b[k]) for k in KEYS), (extra, stop)
            assert a["eta"] == b["eta"] and a["k"] == b["k"] and a["attempts"] == stop
            n1 = [x.kernel_times()[2] for x in (p, q)]
            assert n1[0] - n0[0] >= 2 * 36 > n1[1] - n0[1]
'''


@pytest.mark.parametrize("start", [True, False])
@pytest.mark.parametrize("case", ["words", "words/mixed", "barriers", "barriers/mixed", "far"])
def test_period_that_cannot_be_resident_runs_stepped_with_the_same_bits(case, start):
    _run(f"start = {start}" + NOT_STARTED, case)


ONE_CTA = r'''
limits(p, refuse=1)
p.solve(0.0, 40)
with lpop.Problem(lp, kernel_timing=1, **options) as q:  # timing selects the two step kernels
    q.solve(0.0, 40)
    a, b = p.get_state(), q.get_state()
    assert all(np.array_equal(a[k], b[k]) for k in KEYS)
'''


def test_one_cta_that_is_refused_takes_the_step_kernels():
    _run(ONE_CTA, "one_cta")


LEGACY_STREAM = r'''
with lpop.Problem(lp, stream=1, **options) as q:  # the legacy default stream, which cannot be captured
    limits(q, refuse=1)
    q.solve(0.0, 128)
    p.solve(0.0, 128)
    a, b = q.get_state(), p.get_state()
    assert all(np.array_equal(a[k], b[k]) for k in KEYS)
'''


def test_stepped_period_on_a_stream_that_cannot_be_captured():
    _run(LEGACY_STREAM, "words")
