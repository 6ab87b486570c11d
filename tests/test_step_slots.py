"""The slots that the steps' counters take in turn (csrc/step_slots.cuh), built
with the host's compiler: over the whole range of step numbers, the places where
they pass 2^31 and 2^32 included, a step's slot lies inside the arrays, the
slot a step clears is that of the step before, and neither this step nor the
next one counts there."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2208_13770_gb300", "csrc")

SOURCE = """
#include "step_slots.cuh"
extern "C" {
int slots() { return lvb::kStepSlots; }
int slot_after(unsigned long long done) { return lvb::step_slot(lvb::next_step((unsigned)done)); }
int spent(int slot) { return lvb::spent_slot(slot); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    src, so = str(d / "slots.cpp"), str(d / "slots.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-shared", "-fPIC", "-O2", "-std=c++17", "-I", CSRC, "-o", so, src],
                   check=True)
    out = ctypes.CDLL(so)
    out.slot_after.argtypes = [ctypes.c_ulonglong]
    return out


@pytest.mark.parametrize("around", [3, 1 << 31, 1 << 32, 3 << 31, 1 << 40])
def test_turn_goes_on_over_every_wrap(lib, around):
    for k in range(around - 3, around + 6):
        s = lib.slot_after(k)
        assert 0 <= s < lib.slots()
        if k == 0:
            continue
        before, after = lib.slot_after(k - 1), lib.slot_after(k + 1)
        assert lib.spent(s) == before
        assert before not in (s, after) and s != after
