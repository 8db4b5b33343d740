"""Rules that choose the form of a launch, as plain functions of sizes (no GPU)."""
import ctypes as C
import os
import re

import pytest

from paper_2604_10235_b200 import binding, build


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


FULL = (148, 148, 132, 120), (296, 296, 284, 264)


def _shape(items, seqs=1, hkv=8, chunk=1, fused=1, room=FULL):
    one, two = ((C.c_int * 4)(*r) for r in room)
    cluster, threads = C.c_int(), C.c_int()
    binding.load_library().ccx_select_shape(items, seqs, hkv, chunk, fused, one, two, C.byref(cluster), C.byref(threads))
    return cluster.value, threads.value


@pytest.mark.parametrize("seqs,hkv", [(1, 1), (1, 8), (8, 8), (32, 8), (64, 32)])
@pytest.mark.parametrize("chunk", [1, 10])
def test_shape_of_the_selection_follows_the_device(seqs, hkv, chunk):
    """Every shape holds its items (32 steps per warp) and uses a width that the device has room for, whatever
    its number of SMs per GPC; items beyond the widest cluster are left to the other kernel."""
    for items in (1, 513, 2048, 16384, 16385, 35784, 65536, 131072, 131073, 262144):
        for room in (FULL, ((148, 148, 0, 0), (296, 296, 0, 0)), ((20, 20, 16, 8), (40, 40, 32, 16))):
            cluster, threads = _shape(items, seqs, hkv, chunk, 1, room)
            if cluster == 0:
                assert items > 32 * 1024 * max(1 << i for i in range(4) if room[0][i])
                continue
            assert cluster in (1, 2, 4, 8) and threads in (512, 1024) and room[0][cluster.bit_length() - 1] > 0
            assert cluster * threads * 32 >= items
    assert _shape(262145, seqs, hkv, chunk)[0] == 0 and _shape(0, seqs, hkv, chunk) == (1, 512)


@pytest.mark.parametrize("chunk", [1, 4, 33])
def test_every_shape_of_the_selection_is_one_that_is_chosen(chunk):
    """Each shape that is compiled is the cheapest for some batch on this device, and whatever the device no other is chosen."""
    has = binding.load_library().ccx_select_has_shape
    compiled = {(c, t) for c in (1, 2, 4, 8) for t in (512, 1024) if has(chunk, c, t)}
    sizes = sorted({int(1.07 ** i) for i in range(186)} | {16385, 65537})
    problems = [(1, 1), (1, 8), (2, 8), (5, 4), (8, 8), (19, 8), (32, 8), (64, 32)]
    chosen = {_shape(items, s, h, chunk) for items in sizes for s, h in problems}
    assert chosen - {(0, 0)} == compiled
    for room in (((148, 148, 0, 0), (296, 296, 0, 0)), ((20, 20, 16, 8), (40, 40, 32, 16)), ((132, 132, 132, 132), (264,) * 4),
                 ((16, 64, 128, 144), (16, 64, 200, 280))):
        assert {_shape(items, s, h, chunk, 1, room) for items in sizes for s, h in problems} - {(0, 0)} <= compiled


def test_a_wave_of_wide_clusters_is_as_wide_as_the_device():
    """Fourteen problems of 65536 items: 112 CTAs in clusters of eight are one wave where 120 run at a time and
    two where 96 do, and then narrower clusters are cheaper."""
    assert _shape(65536, 7, 2)[0] == 8
    assert _shape(65536, 7, 2, room=((148, 148, 128, 96), (296, 296, 256, 192)))[0] == 4


@pytest.mark.parametrize("items", [1, 40])
def test_row_statistics_cost_the_ring_of_k_tiles_nothing(items):
    """As many tiles of 32 KB as Q, 18 KB of hand-over buffers and 2 KB of statistics leave of 227 KB, in whichever of its two forms
    pass 2 has the statistics."""
    ring = binding.load_library().ccx_score_ring
    for rows in range(16, 513, 16):
        one, two, added, smem = C.c_int(), C.c_int(), C.c_int(), C.c_size_t()
        ring(rows, items * 148, 148, C.byref(one), C.byref(two), C.byref(added), C.byref(smem))
        least = min(6, (232448 - 1024 - 20480 - 256 * rows) // 32768)
        assert one.value >= two.value >= least >= 2, rows
        assert one.value <= 6 and smem.value <= 232448
        assert items == 40 or not added.value


def test_no_switch_of_a_build_changes_a_kernel():
    """What is tested is what is built: no constant of the sources can be set from the compiler's command line."""
    for name in os.listdir(build.CSRC):
        with open(os.path.join(build.CSRC, name)) as f:
            assert not re.search(r"^\s*#\s*(ifn?def|if|elif)\b", f.read(), re.M), name
