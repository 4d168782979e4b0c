"""Index and time arithmetic of the attention kernel that a launch would take hours to bring to its ends: the kernel's own functions
(csrc/attn_common.cuh), compiled for the host and compared with plain 64-bit arithmetic.  Needs nvcc, no GPU."""
import os
import subprocess

import pytest

from paper_2604_03260_b200 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "attn_common.cuh"
using namespace focus;

static void check(bool ok, const char* what, long long a, long long b) {
    if (!ok) { std::printf("%s at %lld, %lld\n", what, a, b); std::exit(1); }
}

// use `k` of a ring of N slots is in slot k % N, and its full barrier completes the phase of parity (k / N) & 1
template <int N> static void ring() {
    RingAt<N> at;
    for (long long k = 0; k < 100; ++k, at.next()) check(at.slot == k % N && at.phase == ((k / N) & 1), "ring", N, k);
    for (long long start : {(1ll << 31) - 50, (1ll << 32) - 50, (1ll << 33) - 50, (1ll << 40) - 50}) {
        at.slot = (uint32_t)(start % N);
        at.phase = (uint32_t)((start / N) & 1);
        for (long long k = start; k < start + 100; ++k, at.next()) check(at.slot == k % N && at.phase == ((k / N) & 1), "ring", N, k);
    }
    check(sizeof(at) == 8, "a slot and a phase", N, sizeof(at));
}

int main(int, char** argv) {
    switch (std::atoi(argv[1])) {
        case 0: ring<2>(); ring<3>(); ring<4>(); ring<5>(); ring<6>(); ring<8>(); break;
        default: return 2;
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("attn_host")
    (d / "host.cu").write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, str(d / "host.cu"), "-o", str(d / "host")],
                   check=True)
    return lambda which: subprocess.run([str(d / "host"), str(which)], capture_output=True, text=True)


def test_places_in_a_ring_never_run_out(program):
    out = program(0)
    assert out.returncode == 0, out.stdout
    text = open(os.path.join(build.CSRC, "attn_sm100.cu")).read()
    assert "RingAt<C::NSTAGE>" in text and "% C::NSTAGE" not in text and "% C::NINFO" not in text
