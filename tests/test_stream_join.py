"""The fork and join of side streams (fork_join of shtb_internal.h), on the CPU
with recorded stand-ins for the two runtime calls: every forked stream is joined
to the caller's, in success and after a launch that fails."""
import os
import shutil
import subprocess

import pytest

from paper_1110_4874_gb300 import build

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>
#include "shtb_internal.h"

static std::vector<std::string> calls;
static int fail_wait;

int shtb_fail(int code, const std::string &) { return code; }
extern "C" const char *cudaGetErrorString(cudaError_t) { return "stand-in"; }
static std::string name(const void *p) { return std::to_string((long)p); }
extern "C" cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    calls.push_back("record " + name(e) + " on " + name(s));
    return cudaSuccess;
}
extern "C" cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    if (fail_wait && --fail_wait == 0) return cudaErrorInvalidValue;
    calls.push_back(name(s) + " waits for " + name(e));
    return cudaSuccess;
}

// n side streams 1 .. n, events 100 ..; launch number `bad` fails with -77
int main(int, char **argv)
{
    const int n = atoi(argv[1]), bad = atoi(argv[2]);
    fail_wait = atoi(argv[3]);
    std::vector<cudaStream_t> side;
    std::vector<cudaEvent_t> ev;
    for (long i = 0; i < n; ++i) side.push_back((cudaStream_t)(1 + i));
    for (long i = 0; i <= n; ++i) ev.push_back((cudaEvent_t)(100 + i));
    const int rc = fork_join((cudaStream_t)50, side.data(), ev.data(), n, [&] {
        for (int i = 0; i <= n; ++i) {
            if (i == bad) return -77;
            calls.push_back("launch " + std::to_string(i));
        }
        return 0;
    });
    for (auto &c : calls) puts(c.c_str());
    printf("%d\n", rc);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """A program of its own: its stand-ins must not meet a CUDA runtime."""
    if not shutil.which("g++") or not os.path.isdir(build._cuda_include()):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("join")
    src, exe = d / "join.cpp", d / "join"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-o", str(exe), str(src), "-I", build.CSRC, "-I", build.INCLUDE,
                    "-I", build._cuda_include(), "-ldl"], check=True)

    def call(n, bad=-1, bad_wait=0):
        out = subprocess.run([str(exe), str(n), str(bad), str(bad_wait)], check=True, capture_output=True, text=True)
        lines = out.stdout.split("\n")[:-1]
        return lines[:-1], int(lines[-1])
    return call


@pytest.mark.parametrize("n", [0, 1, 2, 7])
def test_streams_are_joined_whatever_launch_fails(run, n):
    fork = ["record 100 on 50"] + [f"{i} waits for 100" for i in range(1, n + 1)]
    join = [c for i in range(1, n + 1) for c in (f"record {100 + i} on {i}", f"50 waits for {100 + i}")]
    for bad in range(-1, n + 1):
        calls, rc = run(n, bad)
        launched = n + 1 if bad < 0 else bad
        assert rc == (0 if bad < 0 else -77)
        assert calls == fork + [f"launch {i}" for i in range(launched)] + join


def test_a_fork_that_fails_joins_what_it_forked(run):
    calls, rc = run(3, bad_wait=2)
    assert rc != 0
    assert calls[:2] == ["record 100 on 50", "1 waits for 100"]
    assert "50 waits for 101" in calls and not any(c.startswith("launch") for c in calls)
