"""The scratch of a batch plan's split classes (csrc/host_sched.h), checked on
the host against an allocator of limited capacity: large waves where memory
allows, every stream back to the plans' own waves as soon as one piece fails,
and nothing left behind when even those do not fit."""
import os
import random
import shutil
import subprocess

import pytest

from conftest import ROOT

MB = 1 << 20


@pytest.fixture(scope="module")
def scratch(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("bs") / "batch_scratch_harness")
    subprocess.check_call([cxx, "-O2", "-std=c++17", os.path.join(ROOT, "tests", "batch_scratch_harness.cpp"), "-o", exe])

    def run(capacity, streams, classes):
        """(fits, bytes still allocated, waves, bytes per stream)"""
        text = f"{capacity} {streams} {len(classes)}\n" + "".join(f"{s} {p} {n} {w}\n" for s, p, n, w in classes)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
        k = 2 + len(classes)
        return bool(int(out[0])), int(out[1]), [int(x) for x in out[2:k]], [int(x) for x in out[k:]]
    return run


def test_one_wave_where_memory_allows(scratch):
    # 143 pairs of 2^19 32-bit words: one wave of 572 MB instead of waves of 64 pairs
    assert scratch(8 << 30, 2, [(1, 4 * MB, 143, 64)]) == (True, 572 * MB, [143], [0, 572 * MB])
    # above 1 GB a wave is cut there; classes of a stream share its piece
    assert scratch(8 << 30, 2, [(1, 4 * MB, 1000, 64), (1, MB, 300, 256)]) == (True, 1024 * MB, [256, 300], [0, 1024 * MB])


def test_short_memory_shrinks_every_stream(scratch):
    classes = [(1, 4 * MB, 1000, 64), (2, 4 * MB, 70, 64)]
    # 1 GB for the first stream would leave 76 MB where the second needs 256 MB
    assert scratch(1100 * MB, 3, classes) == (True, 512 * MB, [64, 64], [0, 256 * MB, 256 * MB])
    assert scratch(512 * MB, 3, classes)[0]
    assert scratch(512 * MB - 1, 3, classes)[:2] == (False, 0)


def test_fits_whenever_the_plans_own_waves_do(scratch):
    rng = random.Random(5)
    for _ in range(200):
        streams = rng.randint(1, 3)
        classes = [(rng.randrange(streams), rng.choice([1, 2, 4]) * MB, rng.randint(1, 2000), rng.choice([1, 64, 256]))
                   for _ in range(rng.randint(0, 5))]
        least = sum(max([min(w, n) * p for s, p, n, w in classes if s == k], default=0) for k in range(streams))
        capacity = rng.choice([least - 1, least, least + 100 * MB, 1 << 31, 8 << 30])
        fits, held, waves, pieces = scratch(max(capacity, 0), streams, classes)
        assert fits == (least <= max(capacity, 0))
        assert held == (sum(pieces) if fits else 0) and held <= max(capacity, 0)
        for (s, p, n, w), wave in zip(classes, waves):
            if fits:
                assert min(w, n) <= wave <= n and wave * p <= pieces[s] <= max(1 << 30, max(min(b, c) * a for t, a, c, b in classes if t == s))
