"""Size and order of a call's slabs on two streams (csrc/ef_slabs.h), compiled with the host compiler."""
import itertools
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_12416_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ef_slabs.h"
int main(int argc, char** argv) {
    if (argc == 7) {  // nb, t, sms, segment, seg_bytes, slab_bytes
        printf("%ld\n", (long)ef::chunk_trajectories(atoll(argv[1]), atoll(argv[2]), atoll(argv[3]), atoll(argv[4]), atoll(argv[5]),
                                                     atoll(argv[6])));
        return 0;
    }
    if (argc > 7) {  // nb, n_chunks, n_seg, item, image, budget, sms, blocks
        const int64_t nb = atoll(argv[1]), nc = atoll(argv[2]);
        const int64_t slab = ef::slab_items_of(nb, nc, atoll(argv[3]), atoll(argv[4]), atoll(argv[5]), atoll(argv[6]), atoll(argv[7]),
                                               atof(argv[8]));
        printf("%ld %ld\n", (long)slab, (long)ef::slab_images(nb, slab, nc));
        return 0;
    }
    const long items = atol(argv[1]), slab = atol(argv[2]), two = atol(argv[3]), bad = atol(argv[4]);
    long n = 0;
    const auto step = [&](const char* what) {
        printf("%s ", what);
        return (int)(bad == ++n ? 100 + n : 0);
    };
    const int e = ef::for_slabs<int>(items, slab, two, [&] { return step("fork"); }, [&] { return step("join"); },
        [&](int64_t i0, int64_t k, int turn) {
            printf("%ld+%ld@%d ", (long)i0, (long)k, turn);
            return bad == ++n ? (int)(100 + n) : 0;
        });
    printf("%d\n", e);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("slabs")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    return lambda *a: subprocess.run([str(d / "m"), *map(str, a)], check=True, capture_output=True, text=True).stdout.split()


def test_slabs_cover_the_items_in_turn(run):
    assert run(7, 3, 0, 0) == ["0+3@0", "3+3@0", "6+1@0", "0"]
    assert run(7, 3, 1, 0) == ["fork", "0+3@0", "3+3@1", "6+1@0", "join", "0"]
    assert run(3, 3, 0, 0) == ["0+3@0", "0"]


def test_a_failed_launch_still_joins(run):
    # steps: fork 1, launches 2 .., join last
    assert run(9, 3, 1, 3) == ["fork", "0+3@0", "3+3@1", "join", "103"]
    assert run(9, 3, 1, 2) == ["fork", "0+3@0", "join", "102"]
    assert run(9, 3, 1, 5) == ["fork", "0+3@0", "3+3@1", "6+3@0", "join", "105"]
    assert run(9, 3, 1, 1) == ["fork", "101"]  # nothing is on the side stream yet
    assert run(9, 3, 0, 2) == ["0+3@0", "3+3@0", "102"]


def test_slabs_stay_within_the_budget(run):
    budget, sms = 512 << 20, 152
    seen = set()
    for nb, nc, item, image in itertools.product((1, 7, 300, 1776, 1900, 8192), (1, 3, 12, 1824), (0, 9000, 290_000, 900_000),
                                                 (400, 50_000, 200_000)):
        for blocks in (1e6, 1e10):
            slab, images = map(int, run(nb, nc, 4, item, image, budget, sms, blocks))
            assert 1 <= slab <= nb * nc and slab * item + images * image <= budget
            whole = image + item * nc <= budget - 2 * image
            assert not whole or slab % nc == 0  # whole bitstrings where one fits
            seen.add((whole, slab < nb * nc, blocks >= 1e9 and slab >= 4 * sms))
    assert {s[0] for s in seen} == {True, False} and any(s[1] for s in seen)


def test_partial_sums_of_long_calls(run):
    sms, seg, seg_bytes, slab = 152, 4096, 73_728, 512 << 20  # every trajectory with an entry
    for nb, t in itertools.product((1, 4, 500, 10_000, 1_000_000), (1, 1000, 68_416, 10 ** 6, 2 ** 32)):
        cut, uncut = (int(run(nb, t, sms, seg, b, slab)[0]) for b in (seg_bytes, 0))
        assert cut % 128 == 0 and 128 <= cut <= uncut <= 2 ** 25
        assert nb * -(-t // cut) <= max(2 ** 24, nb * -(-t // min(uncut, 2 ** 23)))
        assert -(-cut // seg) * seg_bytes <= slab // 2 + seg_bytes
        if nb * t <= 2 ** 24 * 3 * seg:  # within that, an item's samples leave room for 12 per SM in a slab
            assert -(-cut // seg) * seg_bytes <= slab // (4 * sms)
