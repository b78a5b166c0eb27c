"""The plan of the streaming kernels' rows (mm_plan.h, compiled for the host):
no more passes of rows than the cell has, and by its own cost of a pass never dearer than rows of
V nodes to a lane in equal chunks that divide the orientations, which packed
rows replaced."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1908_04279_gb300", "csrc")


def cases():
    for tsz in (4, 8):
        for ns in range(1, 129 if tsz == 4 else 65):
            V = (8 if ns % 8 == 0 else 4 if ns % 4 == 0 else 1) if tsz == 4 else 2 - ns % 2
            if ns // V > 32:
                continue
            for nth in [*range(1, 130), 256, 509, 512, 1024]:
                yield nth, ns, tsz, V


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("plan") / "step_plan_host")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-I" + CSRC,
                           os.path.join(HERE, "step_plan_host.cpp"), "-o", exe])
    text = "\n".join(" ".join(map(str, c)) for c in cases())
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    got = [line.split() for line in out.splitlines()]
    return {c: (int(q[0]), int(q[1]), int(q[2]), int(q[3]), float(q[4]), int(q[5]), int(q[6]))
            for c, q in zip(cases(), got)}


def lane_rpp(ns, V):
    seg = 1
    while seg < ns // V:
        seg *= 2
    return 32 // seg


def test_chunks_cost_no_pass(plans):
    for (nth, ns, tsz, V), (packed, rows, chunks, passes, *_) in plans.items():
        rpp = 32 // -(-ns // 8) if packed else lane_rpp(ns, V)
        at = (nth, ns, tsz, V)
        assert rows <= nth and (chunks - 1) * rows < nth <= chunks * rows, at
        assert passes == -(-nth // rpp), at  # no pass is cut short but the last
        assert rows * ns * tsz <= 4096 or rows <= rpp, at
        assert passes == (chunks - 1) * -(-rows // rpp) + -(-(nth - (chunks - 1) * rows) // rpp), at
        # bulk copies wherever a cell is a whole number of 16-byte vectors
        assert nth * ns * tsz % 16 or rows * ns * tsz % 16 == 0, at


def test_no_dearer_than_equal_chunks_of_lanes(plans):
    for (nth, ns, tsz, V), (_, _, _, _, cost, *_) in plans.items():
        if tsz == 4 and V == 1:
            continue  # (one node to a lane costs 3.5 times a packed one)
        c = 1
        while c < nth and (nth % c or nth // c * ns * tsz > 4096):
            c += 1
        passes = c * -(-(nth // c) // lane_rpp(ns, V))
        before = passes * (V if tsz == 4 else 36.0 if V == 2 else 23.0)
        assert cost <= before * (1 + 1e-12), (nth, ns, tsz, V)


# a substep of the resident kernel over one of the streaming kernel, as timed on a
# GB300 in calls of 16, by orientations, nodes and MB of Mb
TIMED = {(8, 64): {245: 0.62}, (16, 16): {180: 0.54}, (24, 64): {245: 0.95},
         (32, 32): {80: 0.67, 140: 0.83, 245: 0.93}, (32, 64): {245: 0.99}, (32, 31): {450: 0.98},
         (24, 30): {450: 0.74}, (40, 16): {80: 0.86, 140: 1.02, 245: 1.09}, (40, 20): {200: 0.99},
         (48, 16): {80: 0.89, 140: 1.10, 245: 1.17}, (48, 32): {80: 0.74, 160: 1.02, 245: 1.10},
         (64, 16): {60: 0.96, 140: 1.13, 245: 1.20}, (64, 32): {80: 0.86, 200: 1.13, 245: 1.12},
         (64, 64): {80: 0.81, 160: 1.05, 245: 1.09}, (64, 8): {80: 0.92, 120: 1.06},
         (64, 24): {120: 0.90, 245: 1.03}, (64, 40): {245: 0.84}, (48, 31): {120: 0.94, 450: 1.06},
         (64, 31): {120: 0.90, 450: 1.09}}


def test_resident_launch_where_it_was_timed_faster(plans):
    by = {(nth, ns): q[5:] for (nth, ns, tsz, _), q in plans.items() if tsz == 4}
    for (nth, ns), timed in TIMED.items():
        for mb, ratio in timed.items():
            assert (mb << 20 <= by[nth, ns][1]) == (ratio < 1.0), (nth, ns, mb)
    # two substeps: half of the bytes (151 MB of 32 x 32 1.08, 67 MB of 16 x 16 0.65)
    assert by[32, 32][0] < 151 << 20 and by[16, 16][0] > 67 << 20
