"""Resident check periods (csrc/resident.cu): problems held in the shared memory
of one CTA, of several CTAs that exchange words, and of several with grid
barriers (a row or column of more than 128 entries), with long rows cut into
segments and with one side's entries in global memory.

* 40 attempts (online updates included) against the oracle within 1e-10 and
  against the two-kernel path (which kernel timing selects) within 1e-10: the
  free-running bar of the parity tests, which holds for 60 attempts.
* The same attempts split over several lp_solve calls give the same bits: a
  launch takes up exactly the state that the last one left.
* Several problems at a time from host threads, each with the result it has
  alone.
"""
import threading

import numpy as np
import pytest

import lpgen
import oracle
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu

CASES = {
    "one_cta": (lambda: lpgen.tiny_random(3), dict(alpha=1e-3, phi=3)),
    "one_cta_plain": (lambda: lpgen.mixed_small(2), dict(mode="plain", alpha=1e-2, phi=1)),
    "words": (lambda: lpgen.batch_member(9, 701, 1_753), dict(alpha=1e-3, phi=5)),
    "words_transport": (lambda: lpgen.transport(1, 1_501, 1_499, 12_007), dict(alpha=1e-4, phi=20)),
    "barriers_wide_rows": (lambda: lpgen.row_length_mix(2), dict(alpha=1e-3, phi=7)),
    # a row of 4,097..11,000 entries of A and of A^T: segments on both sides
    "barriers_segments": (lambda: lpgen.long_rows(2), dict(alpha=1e-3, phi=20)),
    # too large for shared memory with both copies of the matrix: one side read from global memory
    "one_side_far": (lambda: lpgen.powerlaw(2, 50_000, 125_000, 800_000), dict(alpha=1e-6, phi=20)),
    "barriers_powerlaw": (lambda: lpgen.powerlaw(1, 6_001, 15_003, 90_000, dmax=5_000), dict(alpha=1e-6, phi=20)),
}
MODE = {"plain": lpop.LP_MODE_PLAIN, "pdlp": lpop.LP_MODE_PDLP}


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


def _options(o):
    return dict(o, mode=MODE[o.get("mode", "pdlp")])


def _run(lp, stops, **options):
    with lpop.Problem(lp, **options) as p:
        for k in stops:
            p.solve(0.0, k)
        return p.get_state()


def _close(a, b, rel=1e-10):
    err = np.linalg.norm(np.asarray(a) - np.asarray(b))
    return err <= rel * np.linalg.norm(b) + 1e-14 * np.sqrt(np.size(b))


@pytest.mark.parametrize("case", sorted(CASES))
def test_attempts_match_the_oracle_and_the_two_kernel_path(case):
    make, o = CASES[case]
    lp = make()
    ref = {}

    def trace(P, S):
        if S.attempts == 40:
            ref.update(x=S.x.copy(), y=S.y.copy(), T=S.T.copy(), Sigma=S.Sigma.copy(), ax=S.ax.copy())

    oracle.solve(lp, oracle.Options(**o), tol=0.0, iter_limit=40, trace=trace)
    got = _run(lp, [40], **_options(o))
    two = _run(lp, [40], kernel_timing=1, **_options(o))
    for key in ref:
        assert _close(got[key], ref[key]), f"{case}: {key} against the oracle"
    for key in ("x", "y", "T", "Sigma", "ax", "xbar", "ybar"):
        assert _close(got[key], two[key]), f"{case}: {key} against the two-kernel path"
    assert got["k"] == two["k"] and got["attempts"] == two["attempts"] == 40


@pytest.mark.parametrize("precision", [lpop.LP_PREC_FP64, lpop.LP_PREC_MIXED])
@pytest.mark.parametrize("case", sorted(CASES))
def test_split_runs_give_the_same_bits(case, precision):
    make, o = CASES[case]
    lp = make()
    a = _run(lp, [200], precision=precision, **_options(o))
    b = _run(lp, [1, 8, 64, 65, 130, 200], precision=precision, **_options(o))
    for key in ("x", "y", "T", "Sigma", "ax", "xbar", "ybar", "GT", "GS"):
        assert np.array_equal(a[key], b[key]), f"{case}: {key}"
    assert a["eta"] == b["eta"] and a["k"] == b["k"] and a["restarts"] == b["restarts"]


def test_problems_on_host_threads_and_a_batch_beside_them():
    lps = [CASES[c][0]() for c in ("words", "words_transport", "barriers_wide_rows", "barriers_powerlaw", "words")]
    alone = [_run(lp, [320], alpha=1e-4, phi=20) for lp in lps]
    probs = [lpop.Problem(lp, alpha=1e-4, phi=20) for lp in lps]
    members = [lpop.Problem(lpgen.batch_member(20 + i, 300 + 50 * i, 800), alpha=1e-4, phi=20) for i in range(6)]
    try:
        threads = [threading.Thread(target=p.solve, args=(0.0, 320)) for p in probs]
        with lpop.Batch(members) as b:
            for t in threads:
                t.start()
            for k in range(5):
                b.round(0.0, 64, 320)
            for t in threads:
                t.join()
        for p, ref in zip(probs, alone):
            st = p.get_state()
            assert np.array_equal(st["x"], ref["x"]) and np.array_equal(st["y"], ref["y"])
        for p in members:
            assert p.get_state()["attempts"] == 320
    finally:
        for p in probs + members:
            p.close()
