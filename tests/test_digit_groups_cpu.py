"""The level groups of the digit products, as the sources name them: tcgen05 defines the order of its
instructions into shared TMEM columns only for one accumulator and one shape, so an instruction
writes all columns of its group, and what it multiplies beyond the seven digits has to be zeros."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2003_13245_gb300", "csrc")
ND, NL = 7, 8
FILES = ("zgemm_digits.cu", "qr_tensor.cu")


def read(f):
    with open(os.path.join(CSRC, f)) as fh:
        return fh.read()


def test_one_place_issues_the_products():
    for f in FILES:
        assert "mma_f16(" not in read(f), f
        assert "mma_levels<" in read(f), f


def test_groups_cover_every_digit_pair_once():
    found = [(int(n), int(p, 16)) for f in FILES
             for n, p in re.findall(r"Groups<(\d+), (0x[0-9a-f]+)>", read(f))]
    assert len(found) == 3
    for n, pack in found:
        lo = [(pack >> (4 * g)) & 15 for g in range(n + 1)]
        assert lo[0] == 0 and lo[-1] == NL and sorted(set(lo)) == lo
        lead = max([1] + [min(lo[g + 1] - 1, ND - 1) - lo[g] for g in range(n)])
        pairs = []
        for i in range(ND):
            for g in range(n):
                if i >= lo[g + 1]:
                    assert lo[g + 1] - 1 - i < 0       # left out: no digit of B below zero exists
                    continue
                for level in range(lo[g], lo[g + 1]):
                    j = level - i
                    assert -lead <= j <= ND            # inside the zeros before and behind the run
                    if 0 <= j < ND:
                        pairs.append((i, j))
            if i == 0:
                assert len([g for g in range(n) if lo[g + 1] > 0]) == n   # digit 0 starts all levels
        assert sorted(pairs) == [(i, j) for i in range(ND) for j in range(ND) if i + j < NL]
