"""How a step is ordered on the caller's stream, without a GPU: the step driver linked with a CUDA runtime that only writes
down what it is asked.  Part of a step runs on a stream of the context's own; whether the step succeeds or a call in it
fails, the caller's stream has to wait for that part."""
import ctypes
import os
import subprocess

import pytest

import paper_2510_09103_b200 as A

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_09103_b200", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
MAIN = 7                       # the caller's stream
BUFFERS = [256 * k for k in (1, 2, 3, 4)]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("driver") / "driver.so")
    subprocess.run(["g++", "-std=c++17", "-O0", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", os.path.join(CUDA, "include"), "-x", "c++", os.path.join(CSRC, "ctx.cu"), os.path.join(CSRC, "planner.cpp"),
                    os.path.join(ROOT, "tests", "fake_cuda_runtime.cpp"), "-o", out, "-ldl"], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_begin.argtypes = [ctypes.c_long]
    lib.adapm_workspace_bytes.restype = ctypes.c_size_t
    lib.adapm_workspace_bytes.argtypes = lib.adapm_destroy.argtypes = [ctypes.c_void_p]
    lib.adapm_set_workspace.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t]
    lib.adapm_step.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int64, ctypes.c_void_p]
    return lib


def _context(lib, rows=64, **hp):
    blocks = [A.adapm_block(0, rows, 4096, A.MOM_NONE, 0, A.V_BLOCKMEAN, rows, 0.75, 0.1),     # group sums of its own
              A.adapm_block(rows * 4096, 64, 48, A.MOM_LOWRANK, 3, A.V_BLOCKMEAN, 1, 1.0, 0.1)]
    h = ctypes.c_void_p()
    hpar = A.hparams(grad_dtype=A.GRAD_F32, max_grad_norm=1.0, **hp)
    assert lib.adapm_create((A.adapm_block * 2)(*blocks), 2, ctypes.byref(hpar), ctypes.byref(h)) == 0
    assert lib.adapm_set_workspace(h, BUFFERS[3], lib.adapm_workspace_bytes(h)) == 0
    return h


def _step(lib, h, fail_at):
    """One step; (return code, its log, launches the caller's stream does not wait for, launches that do not wait for it)."""
    lib.fake_begin(fail_at)
    rc = lib.adapm_step(h, *BUFFERS[:3], 1, MAIN)
    log = [(op, int(a), int(b)) for op, a, b in (x.split() for x in lib.fake_log().decode().splitlines())]
    before, seen, event, launches, early = {-1}, {MAIN: {-1}}, {}, set(), []      # -1: the work before the step
    for i, (op, a, b) in enumerate(log):
        if op in ("launch", "memset", "copy"):
            mine = seen.setdefault(a, set())
            if not before <= mine:
                early.append(i)
            mine.add(i)
            launches.add(i)
        elif op == "record":
            event[a] = set(seen.setdefault(b, set()))
        elif op == "wait":
            seen.setdefault(a, set()).update(event.get(b, ()))
        elif op == "sync":                                # the host waited: everything later comes after
            seen[MAIN].update(seen.get(a, ()))
    return rc, log, launches - seen[MAIN], early


@pytest.mark.parametrize("period", [0, 3])
def test_every_way_a_step_can_end_leaves_the_callers_stream_behind_all_of_it(driver, period):
    h = _context(driver, refresh_period=period)
    rc, log, loose, early = _step(driver, h, -1)
    assert rc == 0 and not loose and not early
    assert len({a for op, a, _ in log if op == "launch"}) == 2, "the set is one that forks"
    assert not {"sync", "rebuild"} & {op for op, _, _ in log}
    for n in range(len(log)):
        rc, log_n, loose, early = _step(driver, h, n)
        assert ("failed", 0, 0) in log_n and rc == -4      # ADAPM_ECUDA
        assert not loose and not early, f"call {n} failed: {log_n}"
        assert ("rebuild", 0, 0) in log_n, "the next step must not trust the factors' bf16 copies"
    driver.adapm_destroy(h)


def test_a_set_above_the_limit_stays_on_the_callers_stream(driver):
    h = _context(driver, rows=96 * 1024)                   # 12 bytes per element: 4.8 GB
    rc, log, loose, early = _step(driver, h, -1)
    assert rc == 0 and not loose and not early
    assert {a for op, a, _ in log if op == "launch"} == {MAIN}
    driver.adapm_destroy(h)
