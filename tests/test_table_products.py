"""The limb products counted for strip tables are those of the build that runs:
every entry of a half's table and of a strip's table is made exactly once by the
digit build's chains, sums and copies, and strips of few codes count as chains."""
import numpy as np
import pytest

from paper_2504_14497_gb300 import counts

SPLITS = [(w, k) for w in range(1, 17) for k in range(1, 16 // w + 1)]


@pytest.mark.parametrize("w,k", SPLITS)
def test_halves_are_made_once(w, k):
    s = counts.DigitSplit(1 << 16, w, k)
    assert s.hl + s.hh == w * k and sum(s.bits(d) for d in range(s.ns)) == s.hl
    if s.two or s.nd == 1:
        return                        # the halves are the digits' chains
    chained = sums = 0
    for first, end, pairs in ((0, s.ns, s.pairs[0]), (s.ns, s.nd, s.pairs[1])):
        o = 0
        for d in range(first, end):
            # Of a signed pair's digits 8 and 2^bits - 1 points, 8 and 15 across columns.
            chained += 8 if s.lower(d) else (1 << s.bits(d)) - 1
            if d > first:
                if d == first + 1 and pairs:
                    both, one = s.signed_sums(1 << s.bits(d))
                    sums += 2 * both + one
                else:
                    sums += ((1 << s.bits(d)) - 1) * ((1 << o) - 1)
            o += s.bits(d)
    assert chained + sums == (1 << s.hl) - 1 + (1 << s.hh) - 1


@pytest.mark.parametrize("w,k", SPLITS)
@pytest.mark.parametrize("share", [0.02, 0.4, 1.0])
def test_entries_are_made_once(w, k, share):
    rng = np.random.default_rng(100 * w + k)
    s = counts.DigitSplit(1 << 16, w, k)
    codes = [c for c in range(1, min(1 << (w * k), 4096)) if rng.random() < share]
    none = s.strip_products([], k)
    made = s.strip_products(codes, k) - none
    if s.two:
        both, one = s.signed_sums(1 << s.hh, lambda c: c in set(codes))
        copied = sum(1 for c in codes if (c & 15 == 8 if c >> 4 else c <= 8)) if s.cross else sum(
            1 for c in codes if c & 15 == 0 or c <= 8)
        assert 2 * both + one == len(codes) - copied
        assert made == both * counts.PRODUCTS["affine_pair"] + one * counts.PRODUCTS["affine"]
    elif s.nd > 1:
        low = (1 << s.hl) - 1
        assert made == counts.PRODUCTS["affine"] * sum(1 for c in codes if c & low and c >> s.hl)
    else:
        assert made == 0


def test_build_that_runs():
    rng = np.random.default_rng(5)
    dense = rng.integers(0, 256, (1024, 8))
    by_chains = counts.chain_products(counts.cussen_counts(dense, 8, 1, 16))
    # 22 steps and 255 entries a column: most of them sums that share their factor.
    assert 2 * 16 * 8 * 200 * 356 * 0.7 < counts.table_products(dense, 8, 1, 16) < 0.6 * by_chains
    one = np.full((512, 4), 65535)
    assert counts.table_products(one, 16, 1, 3) == counts.chain_products(counts.cussen_counts(one, 16, 1, 3))
    few_rows = rng.integers(0, 1 << 16, (128, 4))      # halves of 256 entries do not fit the scratch
    assert not counts.DigitSplit(128, 16, 1).fits
    assert counts.table_products(few_rows, 16, 1, 3) == counts.chain_products(counts.cussen_counts(few_rows, 16, 1, 3))


def test_products_of_the_point_formulas():
    # Multiplications and squarings of jac_madd, jac_add and jac_dbl (csrc/ec.cuh).
    for name, mul, sqr in (("madd", 8, 3), ("add", 12, 4), ("dbl", 5, 3), ("affine", 5, 1), ("affine_pair", 7, 2)):
        assert counts.PRODUCTS[name] == 64 * mul + 36 * sqr
