"""The power iteration on matrices with rows of every length.

Plain lp_create estimates ||A~||_2 with a block for each of the longest rows, a
warp for long ones and few lanes for short ones; the no-allocation entry point
knows nothing of the rows.  Both are compared with the same iteration in numpy:
sums of up to 8,192 terms in another order, 1e-11 relative on the norm.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import lpgen
import paper_2506_17650_gb300 as lpop
from oracle.pdhg import splitmix_signs
from paper_2506_17650_gb300 import build as lpbuild

pytestmark = pytest.mark.gpu

CASES = {
    "short_rows": lambda: lpgen.batch_member(1, 900, 2_300),
    "rows_of_every_class": lambda: lpgen.row_length_mix(0),
    "rows_by_blocks": lambda: lpgen.long_rows(0, row_lengths=(4_097, 8_192, 2_049), col_lengths=(4_097, 2_048)),
    "power_law": lambda: lpgen.powerlaw(1, 6_001, 15_003, 90_000, dmax=5_000),
    "mean_of_24": lambda: lpgen.powerlaw(2, 1_500, 1_600, 36_000, dmax=1_200),
    "mean_of_80": lambda: lpgen.powerlaw(3, 900, 1_000, 72_000, dmax=900),
    "dense": lambda: lpgen.tiny_random(0, 150, 160, 150),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


def _numpy(A, iters):
    v = np.full(A.shape[1], 1.0 / np.sqrt(A.shape[1]))
    for _ in range(iters):
        w = A.T @ (A @ v)
        norm = np.linalg.norm(w)
        v = w / norm
    return np.sqrt(norm)


@pytest.mark.parametrize("iters", [1, 7, 60])
@pytest.mark.parametrize("case", sorted(CASES))
def test_norm_matches_the_iteration_in_numpy(case, iters):
    import torch

    lp = CASES[case]()
    with lpop.Problem(lp, mode=lpop.LP_MODE_PLAIN, power_iters=iters) as p:
        dr, dc, sc = p.scaling()
    A = (sp.diags(dr) @ lp.csr() @ sp.diags(dc)).tocsr()
    want = _numpy(A, iters)
    assert sc["norm_est"] == pytest.approx(want, rel=1e-11)
    arrays = []
    for M in (A, A.T.tocsr()):
        M.sort_indices()
        arrays += [torch.tensor(a, device="cuda") for a in (M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data)]
    got = lpop.lp_power_norm_noalloc(lp.m, lp.n, *[a.data_ptr() for a in arrays], iters=iters,
                                     stream=torch.cuda.current_stream().cuda_stream)
    assert got == pytest.approx(want, rel=1e-11)


@pytest.mark.parametrize("iters", [1, 2, 30])
def test_zero_first_product_starts_again_from_the_signs(iters):
    """Rows w (x_i - x_k): the all-ones direction gives exactly zero; ``iters`` rounds from the
    SplitMix64 signs follow, by the caller's column index."""
    import torch

    rng = np.random.default_rng(0)
    m, n = 700, 2_000
    i = rng.integers(0, n, m)
    k = (i + 1 + rng.integers(0, n - 1, m)) % n
    w = rng.uniform(0.5, 2.0, m)
    A = sp.csr_matrix((np.concatenate([w, -w]), (np.tile(np.arange(m), 2), np.concatenate([i, k]))), shape=(m, n))
    A.sort_indices()
    v = splitmix_signs(n) / np.sqrt(n)
    for _ in range(iters):
        z = A.T @ (A @ v)
        norm = np.linalg.norm(z)
        v = z / norm
    arrays = []
    for M in (A, A.T.tocsr()):
        M.sort_indices()
        arrays += [torch.tensor(a, device="cuda") for a in (M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data)]
    got = lpop.lp_power_norm_noalloc(m, n, *[a.data_ptr() for a in arrays], iters=iters,
                                     stream=torch.cuda.current_stream().cuda_stream)
    assert got == pytest.approx(np.sqrt(norm), rel=1e-11)
