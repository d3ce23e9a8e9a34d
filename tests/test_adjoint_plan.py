"""What an adjoint call keeps on the device, and what it falls back to where the device does
not have the memory (csrc/adjoint_plan.h, on the host with an allocator that fails above a
limit)."""
import ctypes
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2409_02964_gb300", "csrc")
KEEP = 512 << 20
ALL, SEGMENT, SUB = 0, 1, 2
SHIM = r"""
#include "adjoint_plan.h"
using namespace lbmv::adj;
// limit: states the device can hold; error: the answer of a try that it cannot (1, or 2: another error)
extern "C" int plan(int dense, int nsteps, int every, long long state_bytes, long long limit, int error, long long* out) {
    Plan p{};
    int tries = 0;
    const int r = allocate_plan(p, dense != 0, nsteps, every, state_bytes, [&](const Plan& q) {
        ++tries;
        return q.seg + q.device_ck <= limit ? 0 : error;
    });
    const long long v[] = {(long long)p.keep, p.K2, p.seg, p.device_ck, p.host_states, tries};
    for (int k = 0; k < 6; ++k) out[k] = v[k];
    return r;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    lib = str(d / "libplan.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, "-o", lib, str(d / "shim.cpp")],
                   check=True)
    fn = ctypes.CDLL(lib).plan
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int,
                   ctypes.c_void_p]

    def call(nsteps, every, state_bytes, limit=1 << 40, dense=False, error=1):
        out = (ctypes.c_longlong * 6)()
        r = fn(int(dense), nsteps, every, state_bytes, limit, error, out)
        return r, tuple(out)

    return call


@pytest.mark.parametrize("nsteps,every", [(1, 1), (1, 7), (2, 1), (80, 20), (80, 21), (60, 60), (60, 100), (4000, 200)])
def test_falls_back_to_less_device_memory(plan, nsteps, every):
    K = min(every, nsteps)
    K2, nck = math.ceil(math.sqrt(K)), (nsteps - 1) // every + 1
    state = max(1, KEEP // nsteps)      # all states fit
    assert plan(nsteps, every, state) == (0, (ALL, K, max(1, nsteps - 1), 0, 1, 1))
    if nsteps - 1 > K:
        assert plan(nsteps, every, state, limit=nsteps - 2) == (0, (SEGMENT, K, K, 0, nck, 2))
    if K > K2:
        r, got = plan(nsteps, every, state, limit=K2)
        assert r == 0 and got[:5] == (SUB, K2, K2, 0, nck + (K - 1) // K2 + 1)
    assert plan(nsteps, every, state, limit=0)[0] == 1                    # not even that
    r, got = plan(nsteps, every, state, limit=0, error=2)                 # another error ends the tries
    assert r == 2 and got[5] == 1


def test_states_beyond_the_limit_are_recomputed(plan):
    assert plan(80, 20, KEEP // 79)[1][0] == ALL
    assert plan(80, 20, KEEP // 79 + 1)[1][0] == SEGMENT
    assert plan(80, 20, KEEP // 20 + 1) == (0, (SUB, 5, 5, 0, 4 + 4, 1))


def test_dense_segments_never_fall_back(plan):
    assert plan(80, 20, 1 << 30, dense=True) == (0, (SEGMENT, 20, 20, 4, 0, 1))
    assert plan(80, 20, 1, limit=3, dense=True)[0] == 1
