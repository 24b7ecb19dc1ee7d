"""The training step's side streams are joined into the caller's stream however
the call ends.  The guard that does it is compiled for the host against a fake of
the CUDA calls, so that a call in the middle of a step can fail."""
import os
import re
import subprocess

import pytest

from paper_2608_02438_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "fork_join.h"

static long fail_at = 0, calls = 0;
static cudaError_t log_call(const char *what, void *a, void *b)
{
    ++calls;
    std::printf("%s %ld %ld\n", what, (long)a, (long)b);
    return calls == fail_at ? cudaErrorUnknown : cudaSuccess;
}
extern "C" {
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return log_call("record", e, s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return log_call("wait", s, e); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return log_call("sync", s, nullptr); }
}

// forks the side stream (2) from the main one (1) and launches on it; `how` 0: joins
// and returns, 1: an error before the join, 2: returns without a fork
static int step(int how)
{
    xp::StreamFork f((cudaStream_t)1, (cudaStream_t)2, (cudaEvent_t)9);
    if (how == 2) return -1;
    if (f.fork((cudaEvent_t)5) != cudaSuccess) return -3;
    std::printf("launch 2\n");
    if (how == 1) return -3;
    return f.join() == cudaSuccess ? 0 : -3;
}

int main(int, char **v)
{
    fail_at = std::atol(v[2]);
    std::printf("rc %d\n", step(std::atoi(v[1])));
    return 0;
}
"""
FORK = ["record 5 1", "wait 2 5"]
JOIN = ["record 9 2", "wait 1 9"]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("fork_join")
    (d / "t.cpp").write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-I" + build.CSRC, "-I" + inc, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("how,fail_at,expect", [
    (0, 0, FORK + ["launch 2"] + JOIN + ["rc 0"]),                   # joined once
    (1, 0, FORK + ["launch 2"] + JOIN + ["rc -3"]),                  # an error after the launch: joined too
    (2, 0, ["rc -1"]),                                               # nothing was forked
    (0, 1, ["record 5 1", "rc -3"]),                                 # the fork failed: nothing to join
    (0, 3, FORK + ["launch 2", "record 9 2"] + JOIN + ["rc -3"]),    # the join failed once: tried again
    (1, 3, FORK + ["launch 2", "record 9 2", "sync 2 0", "rc -3"]),  # it cannot be recorded: waited for
])
def test_side_stream_is_joined(program, how, fail_at, expect):
    out = subprocess.run([program, str(how), str(fail_at)], capture_output=True, text=True, check=True).stdout
    assert out.split("\n")[:-1] == expect


def test_training_step_forks_only_by_the_guard():
    with open(os.path.join(build.CSRC, "train_host.cu")) as f:
        src = f.read()
    assert not re.search(r"cudaStreamWaitEvent|cudaEventRecord", src)
    assert len(re.findall(r"_fork\.fork\(", src)) == 4
