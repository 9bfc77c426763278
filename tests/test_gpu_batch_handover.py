"""Members that pass from FP32 to FP64 inside the batched kernel.

The CTA's first thread ends a member's FP32 phase (at refine_tol, after
refine_stall checks, or to certify a tolerance) while other warps have still to
read the state that led there; without a barrier in between they went separate
ways.  Many members of all sizes that pass over in each of the three ways must
end, certified, with the result that each has in a batch of its own.
"""
import numpy as np
import pytest

import lpgen
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


@pytest.mark.parametrize("how", ["certify", "refine_tol", "refine_stall"])
def test_members_hand_over_in_a_batch(how):
    tol = 1e-4 if how == "certify" else 1e-6
    extra = {"certify": {}, "refine_tol": dict(refine_tol=1e-3), "refine_stall": dict(refine_stall=2, refine_tol=0.0)}[how]
    options = dict(alpha=1e-3, phi=20, precision=lpop.LP_PREC_MIXED, **extra)
    sizes = np.floor(10.0 ** np.random.default_rng(1).uniform(1.7, 3.5, size=40)).astype(int)
    lps = [lpgen.batch_member(500 + i, int(m), int(2.5 * m)) for i, m in enumerate(sizes)]
    probs = [lpop.Problem(lp, **options) for lp in lps]
    try:
        with lpop.Batch(probs) as b:
            assert b.solve(tol, 200_000, 128) == len(probs)
        for i in range(0, len(probs), 9):
            with lpop.Problem(lps[i], **options) as one:
                with lpop.Batch([one]) as b:
                    b.solve(tol, 200_000, 128)
                a, m = one.get_state(), probs[i].get_state()
                assert all(np.array_equal(a[k], m[k]) for k in ("x", "y", "T", "Sigma", "ax")), i
                assert a["attempts"] == m["attempts"]
        for p in probs:
            st = p.result(False, False)[2]
            assert st["status"] == lpop.LP_OPTIMAL and max(st["rel_pres"], st["rel_dres"], st["rel_gap"]) <= tol
    finally:
        for p in probs:
            p.close()
