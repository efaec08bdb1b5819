"""Exactness of the complex128 chain's digit products, checked on the host for
every basis size the path accepts (no GPU): the accumulation chunks hold at most
256 nonzero complex terms of a row (512 real ones), and the FP32 sums of the
first four digit levels then stay at or below 2^24.  The split is read from the
kernel source, so a change of it is checked again here."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2012_12228_gb300", "csrc", "chain_oz.cu")


def test_accumulation_chunks_stay_exact():
    s = open(SRC).read()
    KC = int(re.search(r"constexpr int KC = (\d+);", s).group(1))
    CHUNK = int(re.search(r"constexpr int CHUNK_K = (\d+);", s).group(1))
    expr = re.search(r"const int chunks = (.+?);", s).group(1)
    one, rest = re.fullmatch(r"M - 1 <= CHUNK_K \? (1) : (.+)", expr).groups()
    assert "a.kt0 = tiles * q / chunks;" in s and "a.kt1 = tiles * (q + 1) / chunks;" in s
    terms = 0
    for M in range(20, 2048):
        tiles = -(-M // KC)
        chunks = int(one) if M - 1 <= CHUNK else eval(rest.replace("/", "//"), {"tiles": tiles, "KC": KC, "CHUNK_K": CHUNK})
        for q in range(chunks):
            k0, k1 = tiles * q // chunks * KC, min(M, tiles * (q + 1) // chunks * KC)
            # V's diagonal is zero: a row whose diagonal lies in the chunk has a term less
            inside = k0 == 0 and k1 == M
            terms = max(terms, k1 - k0 - (1 if inside else 0))
    assert terms == 256
    # products of level l = i + j: |d_0| <= 128 (V) and 256 (Z), every other digit at most 64
    for level in range(4):
        pairs = [(128 if i == 0 else 64) * (256 if level - i == 0 else 64) for i in range(level + 1)]
        assert 2 * terms * sum(pairs) <= 2 ** 24
