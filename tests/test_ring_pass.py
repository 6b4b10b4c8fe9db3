"""The KVarN streaming decode's ring of shared-memory stages, on the CPU: the
kernel's own rule for passing stages (csrc/ring_pass.h) under random orders of
landing copies, refills and warps, for the rings it is launched with.  A warp that
goes straight to its next block's stage is found out by the same model."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_04263_gb300", "csrc")


def _const(name):
    text = open(os.path.join(CSRC, "stream_common.cuh")).read()
    return int(re.search(rf"constexpr int {name} = (\d+);", text).group(1))


@pytest.fixture(scope="module")
def sim(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("ring") / "ring")
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "ring_pass_sim.cpp")], check=True)

    def run(ns, blocks, head, seeds, rule):
        return subprocess.run([exe] + [str(x) for x in (_const("kNW"), _const("kSB"), ns, blocks, head,
                                                        seeds, rule)],
                              capture_output=True, text=True, timeout=300)
    return run


@pytest.mark.parametrize("ns,blocks,head", [(1, 40, 40), (2, 53, 53), (2, 53, 20), (2, 7, 7),
                                            (2, 64, 12), (3, 61, 30), (5, 90, 33)])
def test_no_stage_is_taken_for_another(sim, ns, blocks, head):
    res = sim(ns, blocks, head, 25, 0)
    assert res.returncode == 0, res.stdout


def test_skipping_stages_is_found_out(sim):
    assert sim(2, 53, 53, 60, 1).returncode == 1
