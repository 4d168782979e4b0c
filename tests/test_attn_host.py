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

// a wait of up to 4 s that is looked at again only `late` after its end has ended, whenever it began and however late that is
static void wait() {
    for (unsigned long long limit : {1000ull, 2000000ull, 1000000000ull, 4000000000ull})
        for (unsigned long long begin : {0ull, 1ull, 4294967295ull, (1ull << 42) - 1000, 1764859000123456789ull}) {
            const uint32_t t0 = wait_ticks(begin) | 1u, l = wait_limit(limit);
            for (unsigned long long late : {4096ull, 1000000ull, 294967296ull, 295000000ull, 300000000ull, 1000000000ull, 4294967296ull, 600000000000ull})
                check(wait_over(t0, wait_ticks(begin + limit + late) | 1u, l), "a wait that has ended", (long long)limit, (long long)late);
            for (int part = 0; part <= 100; ++part)
                check(!wait_over(t0, wait_ticks(begin + limit / 100 * part) | 1u, l), "a wait that has not ended", (long long)limit, part);
        }
}

// the waits of the item queue say which item of the CTA, all others the query block at work
static void status() {
    for (int where = 1; where < 100; ++where)
        check(stalled_work(where, 7, 3) == (where == 50 || where == 51 ? 3 : 7), "status word 2", where, stalled_work(where, 7, 3));
}

// quotients at both sides of every step near the ends of the range and in it
static void divisor() {
    const long long top = 0x7fffffffll;
    auto one = [&](long long d) {
        if (d < 1 || d > top) return;
        const Divisor by((int)d);
        for (long long q : {0ll, 1ll, 2ll, 1000ll, top / d / 2, top / d - 1, top / d})
            for (long long n : {q * d - 1, q * d, q * d + 1, top - q})
                if (n >= 0 && n <= top) check(by.div((int)n) == n / d, "quotient", n, d);
    };
    for (long long d = 1; d < 20000; ++d) one(d);
    for (int l = 14; l <= 31; ++l)
        for (long long e = -40; e <= 40; ++e) { one((1ll << l) + e); one((1ll << l) / 3 + e); one((1ll << l) / 5 * 3 + e); }
}

int main(int, char** argv) {
    switch (std::atoi(argv[1])) {
        case 0: ring<2>(); ring<3>(); ring<4>(); ring<5>(); ring<6>(); ring<8>(); break;
        case 1: wait(); break;
        case 2: status(); break;
        case 3: divisor(); break;
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


def test_a_wait_that_was_not_looked_at_for_long_has_ended(program):
    out = program(1)
    assert out.returncode == 0, out.stdout


def test_a_wait_of_the_item_queue_names_the_item(program):
    out = program(2)
    assert out.returncode == 0, out.stdout
    text = open(os.path.join(build.CSRC, "attn_sm100.cu")).read()
    assert text.count("give_up(p, &ctl, bad, t.A, ord)") == 4               # every role: TMA, MMA, gate operands, softmax


def test_division_by_a_launch_parameter(program):
    out = program(3)
    assert out.returncode == 0, out.stdout
