"""When step runs are replayed from graphs.  The calls into the CUDA runtime are
counted by a small library loaded ahead of it in a child process, so the test
sees what a run does, not how long it takes.

A context's first short call makes no graph (making one costs as much as it
saves over many steps); short graphs appear once their steps have been wanted
often enough, and runs of 32 steps use one at once.  In 3D, kernel timing
interrupts the replay at the sampled steps only."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COUNTER = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
int made = 0, replayed = 0;
static void* runtime(void) { return dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD); }
int cudaGraphLaunch(void* exec, void* stream) {
    static int (*real)(void*, void*);
    if (!real) real = (int (*)(void*, void*))dlsym(runtime(), "cudaGraphLaunch");
    ++replayed;
    return real(exec, stream);
}
int cudaGraphInstantiate(void** exec, void* graph, unsigned long long flags) {
    static int (*real)(void**, void*, unsigned long long);
    if (!real) real = (int (*)(void**, void*, unsigned long long))dlsym(runtime(), "cudaGraphInstantiate");
    ++made;
    return real(exec, graph, flags);
}
"""
CHILD = r"""
import ctypes, json, sys
sys.path.insert(0, sys.argv[1])
from paper_2512_12934_gb300 import lbm
from paper_2512_12934_gb300 import workloads as W
count = ctypes.CDLL(sys.argv[2])

def seen():
    return ctypes.c_int.in_dll(count, "made").value, ctypes.c_int.in_dll(count, "replayed").value

def calls(run, ns):
    out = []
    for n in ns:
        m0, r0 = seen()
        run.step(n)
        run.sync()
        m1, r1 = seen()
        out.append((m1 - m0, r1 - r0))
    return out

def solver(w):
    return lbm.Solver(w.cfg, w.solid, w.rho, w.u)

channel = W.channel(nx=130, ny=30, R=6, xc=40, u_max=0.02, G12=1.4, Gw=(0.3, -0.3))
box = W.laplace(nx=70, ny=50, R=12, G12=1.2)
drop = W.laplace3(n=20, R=5.0, G12=1.2)
res = {"2d": calls(solver(channel), [10] * 4 + [34]),
       "long": calls(solver(channel), [18] * 2),
       "batch": calls(lbm.Batch([solver(channel), solver(box)]), [10] * 4 + [34])}
s = solver(drop)
s.step(17)
for every in (0, 40):
    s.enable_kernel_timing(every)
    t0 = s.diagnostics()["step"]
    s.step(400)
    s.sync()
    res["3d_%d" % every] = (seen()[1], t0, s.kernel_time_split()[2])
print("RESULT " + json.dumps(res))
"""


@pytest.fixture(scope="module")
def result(tmp_path_factory):
    d = tmp_path_factory.mktemp("count")
    src, so = d / "count.c", d / "count.so"
    src.write_text(COUNTER)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so))
    p = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(so)], env=env, capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads([ln for ln in p.stdout.splitlines() if ln.startswith("RESULT ")][-1][7:])


@pytest.mark.parametrize("kind", ["2d", "batch"])
def test_first_short_calls_make_no_graph(result, kind):
    calls = result[kind]
    assert calls[0] == [0, 0]  # 8 of the 10 steps would have been replayed
    assert calls[1] == [1, 1] and calls[2] == [0, 1] and calls[3] == [0, 1]
    assert calls[4] == [1, 1]  # 32 steps at once


def test_a_call_that_wants_a_short_graph_twice_makes_it(result):
    assert result["long"] == [[1, 2], [0, 2]]


def test_3d_timing_interrupts_replay_at_samples_only(result):
    total0, _, _ = result["3d_0"]
    total1, t0, samples = result["3d_40"]
    first = -t0 % 40
    want, s = 0, 0
    while s < 400:  # runs of 16 before the next sample and before the call's last step
        until = (first - s) % 40
        if min(until, 399 - s) >= 16:
            want, s = want + 1, s + 16
        else:
            s += 1
    assert samples == len([q for q in range(400) if (t0 + q) % 40 == 0])
    assert total1 - total0 == want > 0
