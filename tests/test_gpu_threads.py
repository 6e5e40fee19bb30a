"""Host threads that launch one kernel with different amounts of dynamic shared
memory at the same time."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import genesis_inputs as gi

pytestmark = pytest.mark.gpu

INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include")
FOUR = gi.two_line_spec().lines + [(6301.9, 1.0, 0.3), (6302.1, 1.2, 0.5)]  # 12 components: 42 KB of profile slots
FULL = gi.two_line_pattern_spec().lines + [(6302.1, 1.2, 0.5, 2, 1.0, 1, 1.5)]  # more than 16: 52 KB

# Python threads meet too seldom inside a call of a few microseconds, so native
# ones make the calls: four per problem, all on the default stream; the number
# of calls that returned an error.
HAMMER = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "genesis.h"
extern "C" int hammer(decltype(&me_synth) synth, const me_problem *const *pb, const double *params, int n,
                      void *const *out, int nproblems, int reps)
{
    std::atomic<int> bad{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 4 * nproblems; ++k)
        t.emplace_back([=, &bad] {
            for (int i = 0; i < reps; ++i)
                if (synth(pb[k % nproblems], params, nullptr, n, out[k], nullptr) != ME_OK) ++bad;
        });
    for (auto &x : t) x.join();
    return bad;
}
"""


def test_two_sizes_at_once(gpu, tmp_path):
    src, so = tmp_path / "hammer.cpp", tmp_path / "hammer.so"
    src.write_text(HAMMER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", INCLUDE, "-o", str(so), str(src)],
                   check=True)
    n, pbs, want, outs = 4, [], [], []
    p = torch.tensor(gi.draw_params_uniform(n, 1), device="cuda")
    for lines in (FOUR, FULL):
        spec = gi.ProblemSpec(lines=lines, lambda_grid=np.linspace(6301.0, 6303.0, 40))
        pbs.append(gpu.Problem.from_spec(spec, "f64"))
        want.append(gpu.me_synth(pbs[-1], p))
    outs = [torch.zeros_like(want[k % 2]) for k in range(8)]
    torch.cuda.synchronize()
    from paper_1208_0302_gb300 import _lib
    fn = ctypes.cast(_lib.load().me_synth, ctypes.c_void_p)
    problems = (ctypes.c_void_p * 2)(*[ctypes.addressof(pb._s) for pb in pbs])
    pointers = (ctypes.c_void_p * 8)(*[o.data_ptr() for o in outs])
    lib = ctypes.CDLL(str(so))
    lib.hammer.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p,
                           ctypes.c_int, ctypes.c_int]
    bad = lib.hammer(fn, problems, p.data_ptr(), n, pointers, 2, 2000)
    torch.cuda.synchronize()
    assert bad == 0
    for k, o in enumerate(outs):
        assert torch.equal(o, want[k % 2])
