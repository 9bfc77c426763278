"""The two step kernels, which kernel timing selects whatever a problem's size.

Problems that fit on the SMs iterate in resident periods, so the parity, mixed
and bounds tests no longer reach the step kernels, which large problems and
members handed off by a batch run.  The same comparisons, at the same bars, with
``kernel_timing=1``; every run's launch count shows that its attempts took them.
"""
import subprocess
import sys

import numpy as np
import pytest

import lpgen
import oracle
import paper_2506_17650_gb300 as lpop
from paper_2506_17650_gb300 import build as lpbuild
from tests.conftest import ROOT
from tests.test_gpu_bounds import SCRIPT
from tests.test_gpu_parity import (CASES, close, compare_full_state, compare_state, gpu_options, oracle_steps,
                                   oracle_trace, to_lib_state)

pytestmark = pytest.mark.gpu

CHECK = 3  # kernels of a check


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lpbuild.build()
    lpop.load_library()


def _solve(p, stop, attempts):
    n0 = p.kernel_times()[2]
    p.solve(0.0, stop)
    assert 2 * attempts <= p.kernel_times()[2] - n0 <= 2 * attempts + 2 * CHECK


@pytest.mark.parametrize("case", sorted(CASES))
def test_steps_from_the_oracle_state(case):
    make, o = CASES[case]
    lp = make()
    P, states = oracle_steps(lp, o, 100)
    with lpop.Problem(lp, **gpu_options(o, kernel_timing=1)) as p:
        for k in (1, 2, 3, 4, 20, 21, 22, 41, 63, 64, 65, 100):
            p.set_state(to_lib_state(states[k - 1]))
            _solve(p, k, 1)
            compare_full_state(p.get_state(), states[k], f"{case} step {k}", prev=states[k - 1])


@pytest.mark.parametrize("case", sorted(CASES))
def test_free_running_trajectory(case):
    make, o = CASES[case]
    lp = make()
    horizon = 100 if o.mode == "plain" else 60
    stops = [1, 2, 20, 21, 40, horizon]
    ref, P, _ = oracle_trace(lp, o, stops)
    with lpop.Problem(lp, **gpu_options(o, kernel_timing=1)) as p:
        before = 0
        for k in stops:
            _solve(p, k, k - before)
            before = k
            compare_state(p.iterate(), ref[k], f"{case} attempt {k}")


@pytest.mark.parametrize("precision", [lpop.LP_PREC_FP64, lpop.LP_PREC_MIXED])
@pytest.mark.parametrize("case", ["tiny_plain_norm_freq", "mixed_pdlp_adagrad_norm", "rowmix_pdlp", "long_rows_pdlp",
                                  "transport_small_pdlp", "powerlaw_small_pdlp"])
def test_graph_and_direct_launches_agree_bitwise(case, precision):
    make, o = CASES[case]
    lp = make()
    out = []
    for use_graph in (1, 0):
        with lpop.Problem(lp, **gpu_options(o, use_graph=use_graph, kernel_timing=1, precision=precision)) as p:
            _solve(p, 64, 64)
            _solve(p, 192, 128)
            out.append((p.get_state(), p.kernel_times()[1]))
    for key in ("x", "y", "T", "Sigma", "ax", "xbar", "ybar", "eta", "omega", "k"):
        assert np.array_equal(out[0][0][key], out[1][0][key]), key
    assert np.all(out[0][1] == 3 * 8) and np.all(out[1][1] == 0)  # timed samples: three graph replays, or none


@pytest.mark.parametrize("case", ["tiny_plain_norm_freq", "tiny_pdlp_freq", "mixed_pdlp_adagrad", "rowmix_pdlp",
                                  "long_rows_pdlp", "transport_small_pdlp", "powerlaw_small_pdlp"])
def test_fp32_step_from_the_oracle_state(case):
    make, o = CASES[case]
    lp = make()
    P, states = oracle_steps(lp, o, 70)
    with lpop.Problem(lp, **gpu_options(o, kernel_timing=1, precision=lpop.LP_PREC_MIXED)) as p:
        for k in (1, 2, 5, 20, 21, 40, 63, 64, 65, 70):
            p.set_state(to_lib_state(states[k - 1]))
            _solve(p, k, 1)
            g, r = p.get_state(), to_lib_state(states[k])
            for key in ("x", "y", "ax", "T", "Sigma", "xbar", "ybar"):
                ok, err = close(g[key], r[key], 1e-5)
                assert ok, f"{case} step {k}: {key} differs by {err:.3e} (norm {np.linalg.norm(r[key]):.3e})"
            assert g["k"] == r["k"] and g["attempts"] == r["attempts"] and g["restarts"] == r["restarts"]


def test_x_of_the_longest_columns_from_shared_memory():
    """A power-law LP whose A-row grid is full, whose 4,096 longest columns have a quarter of the
    entries, and with enough entries per block: the FP32 kernel holds their x in shared memory."""
    lp = lpgen.powerlaw(3, 360_001, 900_003, 5_600_000)
    o = oracle.Options(alpha=1e-6, phi=2)
    degree = np.sort(np.bincount(lp.col_idx, minlength=lp.n))[::-1]
    assert 4 * degree[:4096].sum() >= lp.nnz >= 2 * 4096 * 4 * 152  # (four blocks on an SM in FP32)
    P, states = oracle_steps(lp, o, 4)
    for precision, bar in ((lpop.LP_PREC_FP64, 1e-12), (lpop.LP_PREC_MIXED, 1e-5)):
        with lpop.Problem(lp, **gpu_options(o, kernel_timing=1, precision=precision)) as p:
            sc = p.scaling()[2]
            assert sc["grid_a"] <= sc["units_a"]  # a full grid
            for k in (1, 2, 3, 4):
                p.set_state(to_lib_state(states[k - 1]))
                _solve(p, k, 1)
                g, r = p.get_state(), to_lib_state(states[k])
                for key in ("x", "y", "ax", "T", "Sigma", "xbar", "ybar"):
                    ok, err = close(g[key], r[key], bar)
                    assert ok, f"step {k}: {key} differs by {err:.3e} (norm {np.linalg.norm(r[key]):.3e})"


def test_checked_build_reads_no_index_out_of_range_and_matches(tmp_path):
    script = SCRIPT.replace("with lpop.Problem(lp, **opts) as p:", "with lpop.Problem(lp, kernel_timing=1, **opts) as p:")
    assert script != SCRIPT
    out = {}
    for name, lib in (("regular", lpbuild.build()), ("checked", lpbuild.build(checked=True))):
        path = str(tmp_path / f"{name}.npz")
        subprocess.run([sys.executable, "-c", script, ROOT, lib, path], check=True, timeout=1800)
        out[name] = dict(np.load(path))
    assert int(out["checked"]["checked"]) == 1 and int(out["checked"]["bad"]) == 0
    for k in out["regular"]:
        assert k == "checked" or np.array_equal(out["regular"][k], out["checked"][k]), k
