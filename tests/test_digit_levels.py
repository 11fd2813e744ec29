"""Sums of the tensor-core commit: what is claimed to be exact is exact, up to
64 reflectors and 16384 rows (host-side restatement in whole numbers).

Pass 1 keeps every pair (digit k of V, digit l of C) in an FP32 accumulator
of its own over 1024 rows, then adds it to the int32 sum of its level k + l;
levels 0 .. 4 and 5 .. 8 are recombined in int64, and the two parts added in
FP64.  Pass 2 adds all pairs of a level into one FP32 accumulator (64
reflectors at most) and recombines the nine levels in int64.  The sizes that
decide this (chunks, segments, digits a tile takes) are read from the kernel's
own constants."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

from test_digit_scheme import digits, ebound

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_05345_gb300", "csrc")
ND, NLV, DMAX = 8, 9, 127
MAX_ROWS, KMAX, STEP = 16384, 64, 16  # rows of the tensor-core form, reflectors, rows per MMA

PROGRAM = r"""
#include <cstdio>
#include "lhdm_kernels.cuh"
using E = lhdm::Engine<lhdm::GridTeam>;
int main() {
  for (int MT = 1; MT <= 4; ++MT) {
    std::printf("%d %d %d", E::p1_groups(MT), E::p1_slots(MT), E::p1_segment(MT));
    for (int mt = 0; mt < MT; ++mt) std::printf(" %d %d", E::tile_digits<8>(mt, MT), E::tile_digits<16>(mt, MT));
    std::printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def consts(tmp_path_factory):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("levels")
    (d / "c.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    CSRC, "-I", os.path.join(ROOT, "include"), str(d / "c.cu"), "-o", str(d / "c")], check=True)
    out = subprocess.run([str(d / "c")], check=True, capture_output=True, text=True).stdout
    rows = [list(map(int, r.split())) for r in out.splitlines()]
    return {MT + 1: dict(groups=r[0], slots=r[1], chunks=r[2], digits={8: r[3::2], 16: r[4::2]}) for MT, r in enumerate(rows)}


def pairs(lam):
    return [(k, lam - k) for k in range(ND) if 0 <= lam - k < ND]


def test_pass1_accumulators_are_exact(consts):
    for c in consts.values():
        rows = c["chunks"] * c["groups"] * 8
        assert DMAX * DMAX * rows <= 1 << 24          # every whole number up to here is an FP32
    # int32 level sums: at most eight pairs on a level
    assert max(len(pairs(lam)) for lam in range(NLV)) * DMAX * DMAX * MAX_ROWS < 1 << 31


@pytest.mark.parametrize("NB", [8, 16])
def test_pass1_tiles_cover_the_levels(consts, NB):
    for MT, c in consts.items():
        KP, have, cols = 16 * MT, set(), 0
        for mt, nl in enumerate(c["digits"][NB]):
            assert nl <= ND and nl * NB % 16 == 0 and nl * NB <= 256  # N of an MMA
            cols += nl * NB
            for mi in range(128 * mt, 128 * mt + 128):
                k, t = mi // KP, mi % KP
                have |= {(k, l, t) for l in range(nl) if k + l < NLV}
        assert cols <= 512  # columns of tensor memory
        assert have == {(k, l, t) for lam in range(NLV) for k, l in pairs(lam) for t in range(KP)}


def pass2_combine(lev, KP):
    """The nine level sums to u, as the kernel's integers go."""
    lq = []
    for l, v in enumerate(lev):
        f = np.float32(v)
        assert int(f) == v  # exact in the accumulator
        if l <= 3 or KP <= 32:
            s = np.float32(f + np.float32(12582912.0))  # 1.5 2^23
            lq.append(int(np.frombuffer(s.tobytes(), np.int32)[0]) - 0x4B400000)
        else:
            lq.append(v)
        assert lq[-1] == v
    two = [lq[0] * 128 + lq[1], lq[2] * 128 + lq[3], lq[4] * 128 + lq[5], lq[6] * 2 + (lq[7] >> 6) + (lq[8] >> 13)]
    assert all(-2**31 <= t < 2**31 for t in two)
    u = (two[0] << 36) + (two[1] << 22) + (two[2] << 8) + two[3]
    assert -2**63 <= u < 2**63
    return u


@pytest.mark.parametrize("KP", [16, 32, 48, 64])
@pytest.mark.parametrize("sign", [1, -1])
def test_pass2_levels_at_their_largest(KP, sign):
    lev = [sign * len(pairs(lam)) * DMAX * DMAX * KP for lam in range(NLV)]
    u = pass2_combine(lev, KP)
    exact = sum(F(v) * F(2) ** (43 - 7 * lam) for lam, v in enumerate(lev))
    assert exact - 2 < u <= exact


def level_sums(a, b):
    """Exact level sums of digit rows a[i][k], b[i][l]."""
    return [sum(x[k] * y[l] for x, y in zip(a, b) for k, l in pairs(lam)) for lam in range(NLV)]


def pass1_levels(a, b, segment):
    """The kernel's: per pair in FP32 by 16-row steps, int32 every `segment` rows."""
    A, B = np.array(a, np.float32), np.array(b, np.float32)
    lev = [0] * NLV
    for s0 in range(0, len(a), segment):
        for lam in range(NLV):
            for k, l in pairs(lam):
                acc = np.float32(0)
                for r in range(s0, min(s0 + segment, len(a)), STEP):
                    e = min(r + STEP, s0 + segment)
                    acc = np.float32(acc + np.float32(np.dot(A[r:e, k].astype(np.float64), B[r:e, l].astype(np.float64))))
                lev[lam] += int(acc)
                assert abs(lev[lam]) < 2**31
    return lev


@pytest.mark.parametrize("MT,rows", [(1, 1024), (2, 1025), (4, 2100)])
def test_pass1_sums_and_recombination(consts, MT, rows):
    segment = consts[MT]["chunks"] * consts[MT]["groups"] * 8
    rng = random.Random(MT)
    for worst in (True, False):
        v = [1.0 - 2.0**-53 if worst else rng.uniform(-1, 1) for _ in range(rows)]
        c = [1.0 - 2.0**-53 if worst else rng.uniform(-1, 1) * 2.0**-rng.randrange(20) for _ in range(rows)]
        a = [digits(x, 56 - ebound(x)) for x in v]  # a row's own scale
        er = [ebound(x) for x in v]
        ec = max(ebound(y) + e for y, e in zip(c, er))
        b = [digits(y, e + 56 - ec) for y, e in zip(c, er)]
        lev = pass1_levels(a, b, segment)
        assert lev == level_sums(a, b)
        hi = lo = 0
        for lam in range(5):
            hi = (hi << 7) + lev[lam]
        for lam in range(5, NLV):
            lo = (lo << 7) + lev[lam]
        assert abs(hi) < 2**63 and abs(lo) < 2**63
        got = math.ldexp(float(hi), ec - 42) + math.ldexp(float(lo), ec - 70)
        exact = sum(F(x) * F(y) for x, y in zip(v, c))
        # 2 L 2^(Ec - 57) of the digits (both roundings and the levels past 8)
        # and three roundings of sums up to L 2^Ec
        assert abs(F(got) - exact) <= F(2 * rows) * F(2) ** (ec - 57) + 3 * F(rows) * F(2) ** (ec - 53)


def test_first_digit_row():
    # whole groups of 8 rows of W, whatever the passive count
    for nP in range(40):
        for kp in range(5, KMAX + 1):
            r0d = kp + ((8 - ((nP + kp) & 7)) & 7)
            assert kp <= r0d < kp + 8 and (nP + r0d) % 8 == 0


@pytest.mark.parametrize("kp,nP", [(33, 3), (48, 0), (64, 5)])
def test_pass2_elements(kp, nP):
    """x - V D'' for random reflectors of very different scales: each element
    within (3 kp + 2) 2^(Er + Ee - 57) of the exact value of its digits'
    operands, and half an ulp of x and of the result."""
    rng = random.Random(kp)
    KP = (kp + 15) & ~15
    ft = [rng.randrange(-30, 30) for _ in range(kp)]
    d = [math.ldexp(rng.uniform(-1, 1), -f - rng.randrange(6)) for f in ft]
    es = [math.ldexp(x, f) for x, f in zip(d, ft)]  # D'' = 2^Ft D'
    ee = max(ebound(x) for x in es)
    de = [digits(x, 56 - ee) for x in es]
    for _ in range(6):
        v = [math.ldexp(rng.uniform(-1, 1), f - rng.randrange(8)) for f in ft]
        vs = [math.ldexp(x, -f) for x, f in zip(v, ft)]
        er = max(ebound(x) for x in vs)
        a = [digits(x, 56 - er) for x in vs]
        u = pass2_combine(level_sums(a, de), KP)
        x0 = rng.uniform(-1, 1)
        got = x0 - math.ldexp(float(u), er + ee - 57)
        exact = F(x0) - sum(F(p) * F(q) for p, q in zip(v, d))
        part = sum(F(p) * F(q) for p, q in zip(v, d))
        tol = F(3 * kp + 2) * F(2) ** (er + ee - 57) + (abs(part) + abs(F(got))) * F(2) ** -53
        assert abs(F(got) - exact) <= tol
