"""The blocks per slot of the fine hull (Sec. II-B-3) and of the clear before it,
computed by the host: a slot fitted closely to its frame gets as many as one with
room to spare, several slots share what the GPU holds, and no slot goes without.
The rules are compiled into a small host program (no GPU needed)."""
import os
import subprocess

import pytest

from paper_1903_11785_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "fvv_internal.h"
int main() {
    fvv::Tuning tu = fvv::default_tuning();
    int th, waves, sms, slots;
    unsigned words;
    long long rows;
    while (std::scanf("%d %d %d %d %u", &th, &waves, &sms, &slots, &words) == 5) {
        if (th == 0) {   // 0, -, SMs, slots, words, rows: the clear
            if (std::scanf("%lld", &rows) != 1) return 1;
            std::printf("%d\n", fvv::clear_blocks(sms, slots, words, rows));
            continue;
        }
        tu.threads[FVV_TUNE_FINE] = th;
        tu.waves[FVV_TUNE_FINE] = waves;
        std::printf("%d\n", fvv::fine_blocks(tu, sms, slots, words));
    }
}
"""


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    d = tmp_path_factory.mktemp("fine_blocks")
    (d / "rule.cu").write_text(PROGRAM)
    subprocess.run([build._nvcc(), "-std=c++17", "-I", build.CSRC, "-o", str(d / "rule"), str(d / "rule.cu")], check=True,
                   capture_output=True)

    def run(rows):
        out = subprocess.run([str(d / "rule")], input="\n".join(" ".join(map(str, r)) for r in rows), text=True,
                             capture_output=True, check=True).stdout.split()
        return [int(x) for x in out]

    return run


def test_fitted_slots_get_as_many_blocks(blocks):
    sms = 152
    for th in (64, 128, 256):
        for slots in (1, 2, 3, 4, 7, 8, 16, 64, 256):
            resident = sms * 1024 // th
            got = blocks([(th, 16, sms, slots, w) for w in (1, 64, 22302, 44604, 459285, 1 << 23)])
            # a frame of 22,302 words has some 5,500 tiles, more than there are warps
            assert got[2] == got[3] == got[4] == got[5]
            # a share of whole rounds of the blocks that the GPU holds, at least one
            rounds = max(1, slots // 8)
            assert all(1 <= b <= max(1, rounds * resident // slots) for b in got)
            # and no fewer, but for a launch that the tuned shape holds smaller
            assert got[2] == max(1, min(rounds * resident // slots, sms * min(16, 16 * slots) // slots))


@pytest.mark.parametrize("slots", [1, 2, 8, 64, 256])
def test_the_clear_has_blocks_for_the_depth_images_too(blocks, slots):
    sms, rows = 152, 16 * 1080
    got = blocks([(0, 0, sms, slots, w, rows) for w in (1, 5000, 75790, 1 << 23)])
    # at least half of the eight blocks per SM that the largest capacity has
    assert got == sorted(got) and got[0] >= min(rows // 8, got[-1] // 2) and got[-1] == max(1, 8 * sms // slots)
    # images of a few rows take no more than the words do
    assert blocks([(0, 0, sms, slots, 1 << 23, 8)]) == [got[-1]]
