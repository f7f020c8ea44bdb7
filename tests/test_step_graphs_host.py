"""Which steps of a call replay a graph, and that the autotuners time none that
builds one (the host code compiled on its own)."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_13769_gb300", "csrc")
SRC = """
#include "lbm_step_graphs.h"
using namespace lbm;
// A body stepped by calls of the given lengths: graphs built in the last call.
extern "C" int built_in_last_call(const long long* calls, int n, int small) {
    bool have[2][2] = {{false, false}, {false, false}}, warm = false, initialized = false;
    int parity = 0, built = 0;
    int64_t steps = 0;
    for (int k = 0; k < n; ++k) {
        built = 0;
        if (!initialized) parity ^= 1;
        initialized = true;
        int64_t left = calls[k], queued = 0;
        auto plain = [&] { ++steps; --left; parity ^= 1; };
        if (!warm && left > 1) {
            plain();
            warm = true;
        }
        while (left > kGraphShort) {
            const int m = next_steps(left, queued, steps, small != 0, have[1][parity], have[0][parity]);
            queued += m;
            if (m == 1) {
                plain();
                continue;
            }
            bool& h = have[m == kGraphChunk][parity];
            built += !h;
            h = true;
            steps += m;
            left -= m;
        }
        while (left > 0) plain();
    }
    return built;
}
// A batch: a graph whenever more than 64 steps are left.
extern "C" int batch_built_in_last_call(const long long* calls, int n) {
    bool have[2] = {false, false}, warm = false;
    int64_t steps = 0;
    int built = 0;
    for (int k = 0; k < n; ++k) {
        built = 0;
        int64_t left = calls[k];
        if (!warm && left > 1) {
            ++steps;
            --left;
            warm = true;
        }
        for (; left > kGraphChunk; left -= kGraphChunk, steps += kGraphChunk) {
            built += !have[steps & 1];
            have[steps & 1] = true;
        }
        steps += left;
    }
    return built;
}
extern "C" long long warm_calls(int which) { return which == 0 ? kWarmFirst : (which == 1 ? kWarmRest : kBatchWarm); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("graphs")
    (d / "g.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fPIC", "-shared", "-I", CSRC, "-o",
                    str(d / "g.so"), str(d / "g.cpp")], check=True)
    L = C.CDLL(str(d / "g.so"))
    L.warm_calls.restype = C.c_longlong
    return L


def _calls(*n):
    return (C.c_longlong * len(n))(*n), len(n)


@pytest.mark.parametrize("small", [0, 1])
def test_a_timed_call_of_the_autotuner_builds_no_graph(host, small):
    warm = host.warm_calls(0), host.warm_calls(1)
    for n in [*range(1, 300), 1000, 4096, 99999, 100000]:
        assert host.built_in_last_call(*_calls(*warm, n), small) == 0, n


def test_a_timed_call_of_the_batch_autotuner_builds_no_graph(host):
    for n in [*range(1, 300), 1000, 4096, 99999, 100000]:
        assert host.batch_built_in_last_call(*_calls(host.warm_calls(2), n)) == 0, n


@pytest.mark.parametrize("small,first,built", [(1, 17, 0), (1, 20, 0), (1, 32, 0), (1, 48, 1), (1, 64, 1), (1, 200, 2),
                                               (0, 20, 0), (0, 33, 0), (0, 34, 1), (0, 200, 2)])
def test_graphs_of_a_first_call(host, small, first, built):
    """A first call's first 16 steps build none."""
    assert host.built_in_last_call(*_calls(first), small) == built


def test_repeated_short_calls_of_a_small_body_replay_a_graph(host):
    assert host.built_in_last_call(*_calls(20, 20), 1) == 1
    assert host.built_in_last_call(*_calls(20, 20, 20), 1) == 0
