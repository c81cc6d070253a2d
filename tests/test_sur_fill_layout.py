"""Layout of the surrogate's training GEMM operands in shared memory
(csrc/bte_sur_kernels.cu): where the asynchronous copies put each element
against where the tensor cores' descriptors look for it, for both operand
orders, with the sizes read from the source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1401_6047_gb300", "csrc",
                   "bte_sur_kernels.cu")
TEXT = open(SRC).read()


def _const(name):
    env = {"GM": 128, "GN": 128, "GK": 64}
    for n, e in re.findall(r"\b(k?G\w+) = ([^,;]+)[,;]", TEXT):
        env.setdefault(n, eval(re.sub(r"\(size_t\)", "", e).replace("/", "//"), {}, env))
        if n == name:
            return env[n]
    raise KeyError(name)


GM, GK, STAGES, THREADS = 128, 64, _const("kGStages"), _const("kGThreads")
CORE, GROUP, TILE, GROUP_MN = _const("kGCore"), _const("kGGroup"), _const("kGTileBytes"), _const("kGGroupMN")


def _fill_rows():
    """load_rows: {byte: (row, first k)} of every 16-byte copy, and each warp's copies."""
    at, warps = {}, []
    for q in range(GM // 8):
        for warp in range(THREADS // 32):
            r, lanes = q * 8 + warp, []
            for lane in range(32):
                d = (lane >> 3) * TILE + (lane & 7) * CORE + (r >> 3) * GROUP + (r & 7) * 16
                assert d not in at
                at[d] = (r, lane * 8)
                lanes.append(d)
            warps.append(lanes)
    return at, warps


def _fill_mn():
    """load_stage_mn: {byte: (first row, k)} of one stage."""
    at, warps = {}, []
    for q in range(4):
        for t in range(THREADS):
            c = t + q * THREADS
            rb, k = c & 15, c >> 4
            d = (k >> 3) * GROUP_MN + rb * CORE + (k & 7) * 16
            assert d not in at
            at[d] = (rb * 8, k)
            if t % 32 == 0:
                warps.append([])
            warps[-1].append(d)
    return at, warps


def test_rows_land_where_the_descriptors_look():
    """K-major: stage, 16 k per MMA, next core matrix along k CORE bytes and
    along the rows GROUP bytes on; a core matrix is 8 rows of 16 bytes (8 k)."""
    at, _ = _fill_rows()
    seen = set()
    for st in range(STAGES):
        for ks in range(GK // 16):
            for kc in range(2):
                for r in range(GM):
                    d = st * TILE + ks * 2 * CORE + kc * CORE + (r // 8) * GROUP + (r % 8) * 16
                    assert at[d] == (r, st * GK + ks * 16 + kc * 8)
                    seen.add(d)
    assert seen == set(at) and max(at) + 16 <= STAGES * TILE


def test_stored_samples_land_where_the_descriptors_look():
    """MN-major: next core matrix along k GROUP_MN bytes and along the rows
    CORE bytes on; a core matrix is 8 k of 16 bytes (8 rows)."""
    at, _ = _fill_mn()
    seen = set()
    for ks in range(GK // 16):
        for kc in range(2):
            for k in range(8):
                for rb in range(GM // 8):
                    d = ks * 2 * GROUP_MN + kc * GROUP_MN + rb * CORE + k * 16
                    assert at[d] == (rb * 8, ks * 16 + kc * 8 + k)
                    seen.add(d)
    assert seen == set(at) and max(at) + 16 <= TILE


@pytest.mark.parametrize("fill", [_fill_rows, _fill_mn])
def test_copies_are_aligned_and_meet_no_bank_twice(fill):
    """Eight lanes of 16 bytes are one pass over the 32 banks."""
    at, warps = fill()
    assert all(d % 16 == 0 for d in at)
    for lanes in warps:
        for q in range(0, 32, 8):
            assert len({d % 128 for d in lanes[q:q + 8]}) == 8
