"""CPU checks of index and counting rules of the CUDA kernels (csrc/hostdev.h),
compiled for the host with g++."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("hd") / "hostdev_layout")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_1604_07651_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "hostdev_layout.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {k: float(v) for k, v in (line.split() for line in out.strip().splitlines())}


def test_arrivals_at_a_split_tile(results):
    """After any number of rounds at a counter, overlapping ones too, the next
    round's last unit is found and no other."""
    assert results["arrival_violations"] == 0


def test_shared_memory_layouts(results):
    """Every FFT length: elements within their pitch and apart, sequences back
    to back, the constant address steps of each pass, and the computed
    positions of the frequencies."""
    # 2^a <= 4096 but 1, which has no pass, 3 2^a <= 6144, 5 2^a <= 5120, 9 2^a <= 2304: 12 + 12 + 11 + 9
    assert results["fft_lengths"] == 44
    assert results["layout_violations"] == 0


def test_dfts_that_skip_zero_inputs(results):
    """First-pass butterflies of every radix, with all inputs and with the
    upper half zero, against the definition: a few roundings of 6e-8 each."""
    assert results["dft_zeros_rel_l2"] < 5e-7
