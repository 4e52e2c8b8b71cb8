"""The extension module between Python and the scoring calls (csrc/kvp_torch.cpp): what a caller sees of threads and errors."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

# A stand-in for libkvp.so whose scoring calls return once another thread has called let_go(), or -6 after five seconds.
STANDIN = r"""
#include <time.h>
#include <unistd.h>
static volatile int inside, gone;
int is_inside(void) { return inside; }
void let_go(void) { gone = 1; }
static int wait_for_it(void)
{
    int i, rc = -6;
    inside = 1;
    for (i = 0; i < 5000 && rc; ++i) { if (gone) rc = 0; else usleep(1000); }
    inside = gone = 0;
    return rc;
}
int kvp_eval() { return wait_for_it(); }
int kvp_eval_noalloc() { return wait_for_it(); }
int kvp_eval_counts() { return wait_for_it(); }
"""
CALLS = r"""
import ctypes, importlib.util, sys, threading, time
import torch
lib = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
spec = importlib.util.spec_from_file_location("_kvp_torch", sys.argv[2])
m = importlib.util.module_from_spec(spec)
spec.loader.exec_module(m)
schedule = torch.zeros((1, 4, 1), dtype=torch.int32, device="cuda")

def other(over):
    while not lib.is_inside() and not over.is_set():
        time.sleep(0.001)
    lib.let_go()

for call in (lambda: m.eval(1, 4, 1, schedule, True, True, 0), lambda: m.eval_counts(1, 4, 1, schedule, 0),
             lambda: m.eval_noalloc(1, 4, 1, schedule, None, schedule, None, None, None, 0)):
    over = threading.Event()
    t = threading.Thread(target=other, args=(over,))
    t.start()
    r = call()
    over.set()
    t.join()
    print("error" if r.__class__ is int and r != 0 else "ok")
"""


def test_other_threads_run_during_a_scoring_call(tmp_path):
    from paper_2508_13231_b200 import build
    src, lib = tmp_path / "standin.c", tmp_path / "libkvp.so"
    src.write_text(STANDIN)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-w", "-Wl,-soname,libkvp.so", str(src), "-o", str(lib)])
    out = subprocess.run([sys.executable, "-c", CALLS, str(lib), build.BINDING], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert out.returncode == 0 and out.stdout.split() == ["ok"] * 3, out.stdout + out.stderr


def test_out_of_memory_is_torchs_exception():
    """The outputs come from torch's allocator: when it has nothing left the call raises what torch.empty would."""
    import torch

    from paper_2508_13231_b200 import kvp
    access = torch.randint(0, 2 ** 16, (32, 1), dtype=torch.int32, device="cuda")
    prob = kvp.Problem(16, 8192, 32, access, 6, 8, 1, 1)
    schedules = torch.zeros((1 << 17, 32, 1), dtype=torch.int32, device="cuda")    # 34 MB of ticks
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction(1e-4)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            prob.eval(schedules)
        with pytest.raises(torch.OutOfMemoryError):
            prob.eval_counts(schedules)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert prob.eval(schedules)["total_ticks"].unique().numel() == 1
