"""lp_solve from several host threads, also beside batch rounds.

Plans that do not fit on the GPU side by side run stepped (or take turns, when
there are two); a solve's result is bitwise the one it has alone, whatever
runs beside it.
"""
import threading

import numpy as np
import pytest

import lpgen
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "T", "Sigma", "ax", "xbar", "ybar")
ATTEMPTS = 640
LPS = {
    "words": lambda: lpgen.batch_member(9, 4_001, 10_003),
    "few_ctas": lambda: lpgen.batch_member(8, 400, 1_000),
    "transport": lambda: lpgen.transport(1, 5_003, 5_001, 40_009),
    "wide_rows": lambda: lpgen.row_length_mix(2),
    "segments": lambda: lpgen.powerlaw(1, 6_001, 15_003, 90_000, dmax=5_000),
    # a column of more than 16,384 entries: the stepped path forms its segments in a launch of their own
    "segments_apart": lambda: lpgen.long_rows(2, m=24_000, n=30_000, row_lengths=(4_097, 20_000), col_lengths=(17_000, 900)),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


@pytest.fixture(scope="module")
def alone():
    out = {}
    for name, make in LPS.items():
        for precision in (lpop.LP_PREC_FP64, lpop.LP_PREC_MIXED):
            lp = make()
            with lpop.Problem(lp, alpha=1e-4, phi=20, precision=precision) as p:
                p.solve(0.0, ATTEMPTS)
                out[name, precision] = lp, p.get_state(), p.kernel_times()[2]
    return out


def _same(p, ref):
    st = p.get_state()
    for key in KEYS:
        assert np.array_equal(st[key], ref[key]), key
    assert st["eta"] == ref["eta"] and st["k"] == ref["k"]


@pytest.mark.parametrize("count", [2, 6, 24])
def test_results_are_those_of_a_solve_alone(alone, count):
    jobs = [key for _ in range(12) for key in alone][:count] if count > 2 else [("words", lpop.LP_PREC_FP64)] * 2
    probs = [lpop.Problem(alone[j][0], alpha=1e-4, phi=20, precision=j[1]) for j in jobs]
    try:
        together = threading.Barrier(count)

        def solve(p):
            together.wait()
            p.solve(0.0, ATTEMPTS)

        threads = [threading.Thread(target=solve, args=(p,)) for p in probs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for p, j in zip(probs, jobs):
            _same(p, alone[j][1])
            # (which ones ran stepped depends on who came first; two take turns)
            assert count > 2 or p.kernel_times()[2] == alone[j][2]
    finally:
        for p in probs:
            p.close()


def test_solve_beside_rounds(alone):
    members = [lpop.Problem(lpgen.batch_member(20 + i, 1_500, 4_000), alpha=1e-4, phi=20) for i in range(3)]
    probs = [(n, lpop.Problem(alone[n, 0][0], alpha=1e-4, phi=20)) for n in ("words", "few_ctas", "segments_apart")]
    try:
        with lpop.Batch(members) as b:
            threads = [threading.Thread(target=p.solve, args=(0.0, ATTEMPTS)) for _, p in probs]
            for t in threads:
                t.start()
            for _ in range(ATTEMPTS // 64):
                b.round(0.0, 64, ATTEMPTS)
            for t in threads:
                t.join()
        for n, p in probs:
            _same(p, alone[n, 0][1])
        for p in members:
            assert p.get_state()["attempts"] == ATTEMPTS
    finally:
        for p in members + [p for _, p in probs]:
            p.close()
