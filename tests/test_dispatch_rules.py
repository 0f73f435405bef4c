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
