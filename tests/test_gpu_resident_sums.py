"""Sums of long rows in the FP32 phase of a problem that fits in one CTA.

A row of more than 2,048 entries is summed in FP32 pieces of at most eight
terms that are added in FP64, as the step kernels sum it.  With all terms of a
row equal and positive, each piece is off by at most eight roundings
(8 u, u = 2^-24) and the sum is rounded once more to FP32 (u); the FP32 copy of
A~ that the test forms may differ from the library's in the last bit where the
FP64 value is at a tie (2 u).  (One FP32 chain of the 65 or 94 equal terms of a
lane is off by up to 22 u.  3,600 entries take several CTAs, which cut the row.)
"""
import numpy as np
import pytest

import lpgen
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


def _line(k, values, c, as_row):
    """One dense row (or column) of ``k`` entries and nothing else, free variables and equality rows."""
    m, n = (1, k) if as_row else (k, 1)
    rp = np.array([0, k]) if as_row else np.arange(k + 1)
    ci = np.arange(k) if as_row else np.zeros(k)
    return lpgen.LP(m=m, n=n, row_ptr=rp.astype(np.int64), col_idx=ci.astype(np.int32), val=np.full(k, values),
                    b=np.zeros(m), c=np.full(n, c), lb=np.full(n, -np.inf), ub=np.full(n, np.inf),
                    sense=np.full(m, lpgen.SENSE_E, np.uint8), name="line")


def _step(lp, **start):
    """One attempt (vanilla step: always taken) from a state with ``start`` in it."""
    with lpop.Problem(lp, mode=lpop.LP_MODE_PLAIN, ruiz_iters=0, precision=lpop.LP_PREC_MIXED) as p:
        dr, dc, _ = p.scaling()
        st = p.get_state()
        st.update(start, initial_check_done=1)
        p.set_state(st)
        p.solve(0.0, 1)
        assert p.kernel_times()[2] <= 1 + 3  # the attempt ran as one resident launch (and the closing check)
        return np.float32(lp.val[0] * dr[0] * dc[0]).astype(np.float64), st, p.get_state()


@pytest.mark.parametrize("k", [2_049, 3_000, 3_600])
@pytest.mark.parametrize("seed", range(12))
def test_row_of_a(seed, k):
    rng = np.random.default_rng(seed)
    lp = _line(k, rng.uniform(0.5, 2.0), -rng.uniform(0.5, 2.0), True)
    a, _, got = _step(lp, eta=1.0, omega=1.0)
    assert np.all(got["x"] == got["x"][0]) and got["x"][0] > 0  # x+ = -c~
    want = a * float(got["x"][0]) * k
    assert abs(got["ax"][0] - want) <= 11 * U * want


@pytest.mark.parametrize("k", [2_049, 3_000, 3_600])
@pytest.mark.parametrize("seed", range(12))
def test_row_of_the_transpose(seed, k):
    rng = np.random.default_rng(100 + seed)
    lp = _line(k, rng.uniform(0.5, 2.0), 0.0, False)
    y = float(np.float32(rng.uniform(0.5, 2.0)))
    a, _, got = _step(lp, eta=1.0, omega=1.0, y=np.full(k, y))
    want = a * y * k  # x+ = 0 - 1 * 1 * (0 - A~^T y): no further rounding
    assert abs(got["x"][0] - want) <= 11 * U * want
