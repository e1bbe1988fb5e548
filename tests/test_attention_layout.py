"""Shared memory of the prefill attention's row exchange, as the library itself computes it: over every group size, cluster size,
token count and CTA, nothing lies over the rows that may still be on their way to a peer, and everything lies inside."""
import ctypes as C

import pytest

from paper_2503_09387_b200 import binding, build


@pytest.fixture(scope="module")
def lib():
    build.build_library()
    return binding.load_library()


def _can_split(lib, D, G, n):
    f = lib._ZN2vs27prefill_attention_can_splitEiii
    f.restype = C.c_bool
    return n == 1 or f(D, G, n)


def _ranges(lib, D, G, n, n_tok, split):
    r = (C.c_int32 * 10)()
    lib._ZN2vs24prefill_attention_rangesEiiiiiPi(D, G, n, n_tok, split, r)
    names = ("rows", "pairs", "staged", "sums")
    return {k: (r[2 * i], r[2 * i + 1]) for i, k in enumerate(names)}, r[8], r[9]


def _meet(a, b):
    return a[0] < b[1] and b[0] < a[1]


@pytest.mark.parametrize("D", [64, 128])
def test_nothing_lies_over_rows_on_their_way(lib, D):
    for G in range(1, 9):
        for n in (n for n in range(1, 9) if _can_split(lib, D, G, n)):
            for n_tok in range(1, 17):
                for split in range(n):
                    r, ring, total = _ranges(lib, D, G, n, n_tok, split)
                    what = (D, G, n, n_tok, split, r)
                    assert all(0 <= b <= e <= total for b, e in r.values()), what
                    assert not any(_meet(r["staged"], r[k]) for k in ("rows", "pairs", "sums")), what
                    assert not _meet(r["rows"], r["pairs"]) and not _meet(r["rows"], r["sums"]), what
                    assert r["rows"][1] <= ring, what                         # the ring may still be in use when they come
                    if n == 1:                                                # no peers: rows leave from registers, only sums have a place
                        assert r["rows"] == r["pairs"] == r["staged"] == (0, 0), what
                        assert r["sums"][1] - r["sums"][0] == 4 * ((G - 1) * 16 + n_tok), what


@pytest.mark.parametrize("D", [64, 128])
def test_every_group_can_be_split(lib, D):
    assert all(_can_split(lib, D, G, n) for G in range(1, 9) for n in (2, 4))
    assert all(_can_split(lib, D, G, 3) for G in range(1, 8))                     # (eight heads: 144 rows)
    assert not any(_can_split(lib, D, G, n) for G in range(1, 9) for n in (5, 7)) # 16 tokens leave the last CTA none
    assert all(_can_split(lib, D, G, 8) for G in range(1, 8 if D == 128 else 9))
