"""Plan of the resident check periods (csrc/resident_plan.cpp), checked on the CPU.

tests/resident_plan_runner.cpp builds the plan of a matrix; the tests check
that every row of A and of A^T belongs to exactly one item, that a CTA's items
take disjoint entries and rows within the sizes its shared memory is carved
for, that long rows are numbered first and without gaps, that the segments of a
row hold its entries in order, each in a word of its own, and that the plan fits
the limits it was given.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

import lpgen
from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2506_17650_gb300", "csrc")
SEG, SEG_KIND, OWN_KIND, LIMIT = 512, 64, 65, 231_000


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
    h = np.frombuffer(raw, np.int64, 15)
    names = ("ok", "nitems", "ncta", "G", "ep", "ed", "rp", "rd", "lp", "ld", "it", "smem", "total", "bytes", "far")
    p = dict(zip(names, (int(x) for x in h)))
    o = 15 * 8
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
    check(plan(runner, tmp_path, lp, esize, sms), lp, case, sms, esize)


def check(p, lp, case, sms, esize):
    assert p["ok"] or case == "powerlaw"  # (40 SMs do not hold it in FP64)
    if not p["ok"]:
        assert lp.nnz * (esize + 4) + 10 * esize * (lp.m + lp.n) > 0.7 * sms * LIMIT
        return
    assert p["G"] == p["ncta"] <= sms and p["smem"] == p["total"] <= LIMIT
    assert p["nitems"] * 24 + 160 * 40 + 8 * 168 * 16 + (lp.n + 2 * lp.m) * 2 * esize <= p["bytes"] + 4 * 256
    if case == "tiny":
        assert p["G"] == 1
    for side, (rp, rows, cap_e, cap_r, cap_l) in enumerate(((p["At_rp"], lp.n, "ep", "rp", "lp"),
                                                            (p["A_rp"], lp.m, "ed", "rd", "ld"))):
        seen = np.zeros(rows, int)
        words, owned = {}, {}
        for c in p["cta"]:
            items = p["items"][c[2 * side]:c[2 * side + 1]]
            assert len(items) <= p["it"]
            near = not p["far"] >> side & 1
            ent_end, vecs, longs, last_rank = 0, [], 0, 0
            for row0, nrows, length, kind, ent, vec in items:
                rank = {SEG_KIND: 0, OWN_KIND: 3, 0: 2}.get(int(kind), 1)
                assert rank >= last_rank
                last_rank = rank
                if kind == SEG_KIND:  # entries length .. length + nrows of the row, a word of its own
                    assert 0 < nrows <= SEG and vec not in words
                    words[int(vec)] = (row0, length, nrows)
                    assert ent == (ent_end if near else rp[row0] + length)
                    ent_end += nrows
                    continue
                lens = np.diff(rp[row0:row0 + nrows + 1])
                seen[row0:row0 + nrows] += 1
                vecs.extend(range(vec, vec + nrows))
                if kind == OWN_KIND:
                    assert nrows == 1 and length <= 160
                    owned[int(row0)] = (int(ent), int(length))
                    longs += 1
                elif kind == 0:
                    assert near and ent == ent_end and nrows <= 32 and lens.max(initial=0) == length <= 48
                    ent_end += 32 * length
                else:
                    assert kind in (2, 4, 8, 16, 32) and nrows <= 32 // kind and length == vec
                    assert ent == ent_end if near else True
                    assert p["G"] == 1 or lens.max(initial=0) <= SEG
                    longs += nrows
                    ent_end += lens.sum()
            assert (ent_end if near else 0) <= p[cap_e] and longs <= p[cap_l]
            assert longs == c[4 + side] and len(vecs) == c[6 + side] <= p[cap_r]
            assert sorted(vecs) == list(range(len(vecs)))
            for row0, nrows, length, kind, _, vec in items:
                if kind not in (0, SEG_KIND):
                    assert vec + nrows <= longs  # the long rows are the first local rows
                if p["G"] == 1:
                    assert vec == row0
        for row, (first, count) in owned.items():  # a row's words hold its entries, in order
            at = 0
            for k in range(first, first + count):
                r, beg, size = words.pop(k)
                assert r == row and beg == at
                at += size
            assert at == rp[row + 1] - rp[row]
        assert not words
        assert np.all(seen == 1)


@pytest.mark.parametrize("case,sms", [("member", 12), ("transport", 10)])
def test_one_side_stays_in_global_memory_when_both_do_not_fit(runner, tmp_path, case, sms):
    lp = CASES[case]()
    p = plan(runner, tmp_path, lp, 8, sms)
    assert p["ok"] and p["far"] in (1, 2) and p["G"] == sms
    check(p, lp, case, sms, 8)


def test_plan_refuses_what_does_not_fit(runner, tmp_path):
    assert plan(runner, tmp_path, lpgen.long_rows(0), 8, 152)["ok"]
    assert not plan(runner, tmp_path, lpgen.transport(0, 2_000, 2_000, 16_000), 8, 4, 60_000)["ok"]
