"""The size rules of csrc/dispatch.cuh, compiled here as plain C++ and compared
with what they stand for."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_02705_gb300", "csrc")


def _rows(tmp_path, body):
    """Lines of numbers that a program with this main() prints."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = tmp_path / "rules.cpp"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "dispatch.cuh"\nusing namespace roam;\nint main() {' + body + "}\n")
    exe = tmp_path / "rules"
    subprocess.run([gxx, "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


def test_tile_runs_are_multiples_of_the_request_and_of_the_tiles_in_flight(tmp_path):
    rows = _rows(tmp_path, "for (int slots : {1, 2, 4, 6}) for (int pad = 0; pad <= 64; pad += 4)"
                           ' printf("%d %d %d\\n", slots, pad, tile_run(pad, slots));')
    assert len(rows) == 4 * 17
    for slots, pad, run in rows:
        assert run > 0 and run % slots == 0, (slots, pad, run)
        if pad == 0:
            assert run == slots
        else:
            assert run % pad == 0 and run <= pad * slots, (slots, pad, run)


def test_the_library_pads_by_that_rule():
    src = open(os.path.join(CSRC, "roam_api.cu")).read()
    assert "cb.group[k] = tile_run(c->tile_pad, " in src


def test_tiles_in_flight_by_samples_per_field_and_per_sm(tmp_path):
    rows = _rows(tmp_path, "for (int W : {32, 64, 128}) for (int sm : {1, 148, 152}) for (int f : {1, 7, 512, 65535})"
                           " for (long long t : {28LL * 128 * f, 16LL * 128 * sm}) for (long long d : {-1LL, 0LL, 1LL})"
                           ' printf("%d %d %d %lld %d\\n", W, sm, f, t + d, tc_slots(W, t + d, f, sm));'
                           ' printf("32 152 1 0 %d\\n32 152 1 %lld %d\\n", tc_slots(32, 0, 1, 152),'
                           " 1LL << 40, tc_slots(32, 1LL << 40, 1, 152));")
    for W, sm, f, n, slots in rows:
        if W == 32:
            assert slots == (6 if n >= 3584 * f and n >= 2048 * sm else 4), (W, sm, f, n, slots)
        else:
            assert slots == (4 if W == 64 else 2)
    assert {r[-1] for r in rows} == {2, 4, 6}


def test_round_samples(tmp_path):
    rows = _rows(tmp_path, "for (long long n : {1LL, 8192LL, 0x7fffffffLL}) for (int R : {1, 15, 16, 17, 1024})"
                           ' printf("%lld %d %lld %lld\\n", n, R, (long long)round_samples(n, R, true),'
                           " (long long)round_samples(n, R, false));")
    for n, R, first, later in rows:
        assert first == n * min(R, 16) and later == first // 8


# voxels, non-empty bricks, voxels per network, us per network from the lists and in the general form (GB300)
ASSIGN = [
    (190528, 2368, 17320, 27.0, 57.7), (190528, 2368, 95264, 71.3, 61.7),
    (1524224, 18944, 3810, 14.5, 62.9), (1524224, 18944, 33135, 49.2, 74.5), (1524224, 18944, 138565, 133.3, 109.0),
    (6193664, 86528, 15484, 34.4, 115.1), (6193664, 86528, 65196, 88.5, 133.1), (6193664, 86528, 269289, 274.2, 211.9),
    (32768, 64, 2048, 12.1, 47.9), (262144, 512, 8192, 29.6, 52.5), (262144, 512, 131072, 76.7, 66.3),
    (2097152, 4096, 33288, 52.9, 81.2), (2097152, 4096, 262144, 187.0, 136.6),
    (16777216, 32768, 65027, 96.4, 244.9), (16777216, 32768, 1048576, 819.4, 529.5),
    (41572, 4096, 8314, 20.2, 54.6), (32978, 20824, 2061, 23.0, 48.8), (32978, 20824, 16489, 101.5, 53.7),
    (326729, 32764, 8168, 26.5, 53.3), (326729, 32764, 36303, 108.5, 68.1),
    (267747, 168116, 2013, 35.3, 49.9), (267747, 168116, 16734, 117.8, 57.9), (267747, 168116, 66936, 376.0, 63.5),
    (1985061, 262026, 8004, 48.9, 71.4), (1985061, 262026, 33084, 148.4, 85.6),
    (99969, 83304, 2040, 30.8, 50.0), (99969, 83304, 16661, 132.7, 59.5),
    (1998122, 1289647, 4995, 150.3, 83.9), (1998122, 1289647, 66604, 511.3, 120.5),
    (19815086, 2097005, 65181, 389.3, 371.6), (19815086, 2097005, 1042899, 3431.2, 915.1),
]


def test_assignment_takes_the_form_measured_faster(tmp_path):
    calls = "".join(f"show({S}, {B}, {per});" for S, B, per, _, _ in ASSIGN)
    rows = _rows(tmp_path, "auto show = [](long long S, long long b, long long per) {"
                           ' printf("%d\\n", (int)assign_from_bricks(S, b, per)); };' + calls)
    for (S, B, per, lists, general), (chosen,) in zip(ASSIGN, rows):
        assert (lists if chosen else general) <= 1.1 * min(lists, general), (S, B, per)
