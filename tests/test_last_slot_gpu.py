"""A candidate whose language would come to the last slot of the largest table (2^32
slots, 0xFFFFFFFF: the number of "not marked") takes the first slot and is marked."""
import os
import subprocess

import pytest

from paper_2305_18575_gb300 import build

pytestmark = pytest.mark.gpu


def test_languages_of_the_last_slot_of_the_largest_table_are_marked(tmp_path):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "last_slot.cu")
    exe = str(tmp_path / "last_slot")
    subprocess.run([build.nvcc(), src, "-o", exe, "-I", build.CSRC, "-O1", "-std=c++17", *build.ARCH], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    if out[0] == "too little memory":
        pytest.skip(out[0])
    assert out[:7] == ["fffffffe", "00000000"] * 3 + ["err 0"]
