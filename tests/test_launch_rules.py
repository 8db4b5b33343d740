"""Rules that choose the form of a launch, as plain functions of sizes (no GPU)."""
import ctypes as C

import pytest

from paper_2604_10235_b200 import binding


@pytest.mark.parametrize("vocab", [5000, 32000, 50257, 151936])
@pytest.mark.parametrize("slots", [444, 396])
def test_split_rows_of_chunk_scoring_never_add_a_wave(vocab, slots):
    rule = binding.load_library().ccx_ppl_split
    whole, parts = C.c_int(), C.c_int()
    for rows in list(range(1, 3001)) + [2 ** 31 - 1]:
        rule(rows, vocab, slots, C.byref(whole), C.byref(parts))
        w, p = whole.value, parts.value
        assert 0 <= w <= rows and 1 <= p <= 8 and w % p == 0
        assert p == 1 or vocab // p >= 8192
        assert -(-(w + (rows - w) * p) // slots) == -(-rows // slots), f"{rows} rows: {w} whole, the others in {p}"
        if rows % slots == 0:
            assert p == 1
        elif rows < slots:                         # few rows: all of them, as far as one wave allows
            assert p == max(1, min(8, slots // rows, vocab // 8192))
