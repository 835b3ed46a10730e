"""Host logic around the recorded cycles and the tuning, against a stand-in for the CUDA runtime (fake_cudart.c): calls are
counted and made to fail, kernels are not run.  Each scenario is a process of its own, which loads libocmg.so with the
stand-in in the place of libcudart.so.13."""
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PREAMBLE = '''
import ctypes as c, importlib.util, os, sys
import numpy as np
spec = importlib.util.spec_from_file_location("_lib", os.path.join(sys.argv[1], "paper_2403_08063_gb300", "_lib.py"))
_lib = importlib.util.module_from_spec(spec)
spec.loader.exec_module(_lib)  # without the package, whose torch brings the real runtime
fake = c.CDLL("libcudart.so.13")
fake.fake_calls.restype = c.c_long
calls = lambda name: fake.fake_calls(name.encode())
fail = lambda name, skip=0: fake.fake_fail(name.encode(), c.c_long(skip))
lib = _lib.load()

def config(n, leaves, problems):
    cfg = _lib.MGConfig(roots=2 if problems == 1 else 1, n=n, n_leaves=len(leaves), interface_flux=1, precision=1, nu1=2,
                        nu2=2, max_coarse=512, inner_cycles=1, n_problems=problems)
    cfg.keep = np.ascontiguousarray(leaves, dtype=np.int32)
    cfg.leaves = cfg.keep.ctypes.data_as(c.POINTER(c.c_int32))
    return cfg

def forest(n=16):
    cfg = config(n, [(0, 0, i, j, k) for k in (0, 1) for j in (0, 1) for i in (0, 1)], 1)
    h = c.c_void_p()
    assert lib.mg_forest_create(c.byref(cfg), c.byref(h)) == 0
    return h

field = np.zeros(1 << 16)
F = field.ctypes.data_as(c.c_void_p)
cycles = lambda h, count: lib.mg_vcycle(h, F, count, None)

def tail_of(h):
    level = c.c_int32()
    assert lib.mg_get_tail(h, c.byref(level)) == 0
    return level.value

def shape(h, threads):
    return lib.mg_set_smoother_shape(h, 0, (c.c_int32 * 5)(1, 1, threads, 0, 0))
'''


@pytest.fixture(scope="module")
def scenario(tmp_path_factory):
    from paper_2403_08063_gb300.build import build
    build()
    gcc = shutil.which("gcc")
    if not gcc:
        pytest.skip("no gcc")
    where = tmp_path_factory.mktemp("fake")
    versions = where / "versions.map"
    versions.write_text("libcudart.so.13 { global: *; };")
    subprocess.run([gcc, "-shared", "-fPIC", "-O1", "-w", "-Wl,-soname,libcudart.so.13", f"-Wl,--version-script,{versions}",
                    os.path.join(HERE, "fake_cudart.c"), "-o", str(where / "libcudart.so.13")], check=True)

    def run(body):
        r = subprocess.run([sys.executable, "-c", PREAMBLE + body, ROOT], capture_output=True, text=True, timeout=300,
                           env={**os.environ, "LD_LIBRARY_PATH": str(where)})
        assert r.returncode == 0, r.stdout + r.stderr
    return run


def test_a_cycle_is_recorded_at_its_second_run_and_replayed(scenario):
    scenario('''
h = forest()
assert lib.mg_set_rhs(h, F, None) == 0
b, g = calls("cudaStreamBeginCapture"), calls("cudaGraphLaunch")
assert cycles(h, 1) == 0 and calls("cudaStreamBeginCapture") == b
assert cycles(h, 3) == 0 and calls("cudaStreamBeginCapture") == b + 1 and calls("cudaGraphLaunch") == g + 3
''')


def test_a_new_shape_or_tail_runs_directly_before_it_is_recorded(scenario):
    """The direct run loads the kernels, which a recording does not allow."""
    scenario('''
h = forest()
assert lib.mg_set_rhs(h, F, None) == 0 and cycles(h, 3) == 0
for change in (lambda: shape(h, 512), lambda: lib.mg_set_tail(h, 1), lambda: lib.mg_set_tail(h, -1)):
    assert change() == 0
    b, g = calls("cudaStreamBeginCapture"), calls("cudaGraphLaunch")
    assert cycles(h, 1) == 0 and calls("cudaStreamBeginCapture") == b and calls("cudaGraphLaunch") == g
    assert cycles(h, 2) == 0 and calls("cudaStreamBeginCapture") == b + 1 and calls("cudaGraphLaunch") == g + 2
''')


def test_a_failed_recording_is_tried_again_after_the_next_change(scenario):
    scenario('''
h = forest()
assert lib.mg_set_rhs(h, F, None) == 0 and cycles(h, 1) == 0
g = calls("cudaGraphLaunch")
fail("cudaGraphInstantiate")
assert cycles(h, 3) == 0 and calls("cudaGraphLaunch") == g  # launched one by one
assert shape(h, 512) == 0
assert cycles(h, 3) == 0 and calls("cudaGraphLaunch") == g + 2
''')


def test_a_launch_that_fails_in_a_recording_is_not_left_out_of_the_replays(scenario):
    scenario('''
h = forest()
assert lib.mg_set_rhs(h, F, None) == 0
n = calls("launch")
assert cycles(h, 1) == 0
n = calls("launch") - n
g = calls("cudaGraphLaunch")
fail("launch", n // 2)  # most launches of the call are the cycle's
assert cycles(h, 1) == 0 and calls("cudaGraphLaunch") == g
''')


def test_a_failure_while_the_tail_is_tuned_leaves_it_off(scenario):
    scenario('''
h = forest()
fail("cudaGraphLaunch", 9)  # seven per candidate: the first tail's
assert lib.mg_set_rhs(h, F, None) == 5 and tail_of(h) == -1
fake.cudaGetLastError()  # the runtime keeps an error until it is read
g = calls("cudaGraphLaunch")
assert lib.mg_set_rhs(h, F, None) == 0 and calls("cudaGraphLaunch") == g + 21  # tuned now: off and two tails
''')


def test_a_batch_that_changes_a_groups_tail_drops_its_recorded_cycle(scenario):
    scenario('''
cfg = config(8, [(0, 0, 0, 0, 0), (1, 0, 0, 0, 0)], 2)
B = c.c_void_p()
assert lib.mg_batch_create(c.byref(cfg), (c.c_int32 * 2)(8, 16), c.byref(B)) == 0
h = c.c_void_p(lib.mg_batch_group(B, 1))
assert lib.mg_set_tail(h, 0) == 0 and lib.mg_batch_set_rhs(B, F, None) == 0
assert lib.mg_set_tail(h, 1) == 0 and cycles(h, 3) == 0
assert lib.mg_batch_set_tail_mode(B, 1) == 0 and tail_of(h) == 0
b, g = calls("cudaStreamBeginCapture"), calls("cudaGraphLaunch")
assert cycles(h, 1) == 0 and calls("cudaGraphLaunch") == g  # not the cycle with the tail from level 1
assert cycles(h, 1) == 0 and calls("cudaStreamBeginCapture") == b + 1
''')
