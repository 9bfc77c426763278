"""Plan of the resident check periods (csrc/resident_plan.cpp), checked on the CPU.

tests/resident_plan_runner.cpp builds the plan of a matrix; the tests check
that every row of A and of A^T belongs to exactly one item, that a CTA's items
take disjoint entries and rows within the sizes its shared memory is carved
for, that a slice's longest row comes first and long rows are numbered without
gaps, and that the plan fits the limits it was given.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

import lpgen
from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2506_17650_gb300", "csrc")
THREADS, WIDE, MAX_ROW, LIMIT = 512, 16, 8192, 231_000


@pytest.fixture(scope="module")
def runner(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("plan") / "resident_plan_runner")
    subprocess.run([gxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC,
                    os.path.join(ROOT, "tests", "resident_plan_runner.cpp"), os.path.join(CSRC, "host_layout.cpp"),
                    os.path.join(CSRC, "resident_plan.cpp"), "-o", out], check=True, capture_output=True)
    return out


def plan(runner, tmp_path, lp, esize, sms, limit=LIMIT):
    src, dst = str(tmp_path / "in.bin"), str(tmp_path / "out.bin")
    with open(src, "wb") as f:
        np.array([lp.m, lp.n, lp.nnz], np.int64).tofile(f)
        lp.row_ptr.astype(np.int64).tofile(f)
        lp.col_idx.astype(np.int32).tofile(f)
        lp.val.astype(np.float64).tofile(f)
    subprocess.run([runner, src, dst, str(esize), str(sms), str(limit)], check=True)
    raw = open(dst, "rb").read()
    h = np.frombuffer(raw, np.int64, 14)
    names = ("ok", "nitems", "ncta", "G", "ep", "ed", "rp", "rd", "lp", "ld", "it", "smem", "total", "bytes")
    p = dict(zip(names, (int(x) for x in h)))
    o = 14 * 8
    p["items"] = np.frombuffer(raw, np.int64, p["nitems"] * 6, o).reshape(-1, 6)
    o += p["nitems"] * 48
    p["cta"] = np.frombuffer(raw, np.int64, p["ncta"] * 8, o).reshape(-1, 8)
    o += p["ncta"] * 64
    p["A_rp"] = np.frombuffer(raw, np.int32, lp.m + 1, o)
    p["At_rp"] = np.frombuffer(raw, np.int32, lp.n + 1, o + 4 * (lp.m + 1))
    return p


CASES = {
    "tiny": lambda: lpgen.tiny_random(0),  # one CTA
    "mixed_small": lambda: lpgen.mixed_small(0),  # empty rows and columns
    "rowmix": lambda: lpgen.row_length_mix(0),  # every row class, empty rows, CTA-wide rows
    "transport": lambda: lpgen.transport(0, 2_001, 1_999, 16_003),
    "member": lambda: lpgen.batch_member(3, 5_001, 12_502),
    "powerlaw": lambda: lpgen.powerlaw(0, 20_000, 50_000, 300_000, dmax=8_000),
}


@pytest.mark.parametrize("esize", [8, 4])
@pytest.mark.parametrize("sms", [152, 40])
@pytest.mark.parametrize("case", sorted(CASES))
def test_plan_covers_every_row_once_and_fits(runner, tmp_path, case, sms, esize):
    lp = CASES[case]()
    p = plan(runner, tmp_path, lp, esize, sms)
    assert p["ok"] or case == "powerlaw"  # (40 SMs do not hold it in FP64)
    if not p["ok"]:
        assert 2 * lp.nnz * (esize + 4) + 10 * esize * (lp.m + lp.n) > 0.7 * sms * LIMIT
        return
    assert p["G"] == p["ncta"] <= sms and p["smem"] == p["total"] <= LIMIT
    assert p["nitems"] * 24 + 160 * 40 + 8 * 168 * 16 + (lp.n + 2 * lp.m) * 2 * esize <= p["bytes"] + 4 * 256
    if case == "tiny":
        assert p["G"] == 1
    for side, (rp, rows, cap_e, cap_r, cap_l) in enumerate(((p["At_rp"], lp.n, "ep", "rp", "lp"),
                                                            (p["A_rp"], lp.m, "ed", "rd", "ld"))):
        seen = np.zeros(rows, int)
        for c in p["cta"]:
            items = p["items"][c[2 * side]:c[2 * side + 1]]
            assert len(items) <= p["it"]
            ent_end, vecs, longs, wide, last_rank = 0, [], 0, 0, 0
            for row0, nrows, length, kind, ent, vec in items:
                lens = np.diff(rp[row0:row0 + nrows + 1])
                seen[row0:row0 + nrows] += 1
                vecs.extend(range(vec, vec + nrows))
                assert ent >= ent_end
                rank = 0 if kind == THREADS else (1 if kind else 2)
                assert rank >= last_rank
                last_rank = rank
                if kind == 0:
                    assert nrows <= 32 and lens.max(initial=0) == length <= 48
                    ent_end = ent + 32 * length
                else:
                    assert kind in (2, 4, 8, 16, 32, THREADS) and nrows <= max(1, 32 // kind) and length == longs
                    assert ent == ent_end  # a long row ends where the next one starts
                    assert lens.sum() <= MAX_ROW
                    longs += nrows
                    wide += kind == THREADS
                    ent_end = ent + lens.sum()
            assert ent_end <= p[cap_e] and longs <= p[cap_l] and wide <= WIDE
            assert longs == c[4 + side] and len(vecs) == c[6 + side]
            if p["G"] == 1:
                assert vecs == [] or set(vecs) == set(range(rows))
                for row0, nrows, length, kind, _, vec in items:
                    assert vec == row0 and (kind == 0 or length == row0)
            else:
                assert vecs == list(range(len(vecs)))  # long rows first, so that a long row's number is its local row
            assert len(vecs) <= p[cap_r]
        assert np.all(seen == 1)


def test_plan_refuses_what_does_not_fit(runner, tmp_path):
    # a column of more entries than a CTA takes, and too little shared memory
    assert not plan(runner, tmp_path, lpgen.long_rows(0), 8, 152)["ok"]
    assert not plan(runner, tmp_path, lpgen.transport(0, 2_000, 2_000, 16_000), 8, 4, 60_000)["ok"]
