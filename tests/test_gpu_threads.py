"""Batches of one context while another thread destroys and retunes contexts of
its own, and batches whose recording as a graph is broken off (the runtime's
answer is a fake's, in a child process): every call succeeds, exactly."""
import os
import subprocess
import sys
import threading
import time
from pathlib import Path

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = Path(__file__).resolve().parent.parent


def _data(seed):
    rng = np.random.default_rng(seed)
    offs = np.array([0, 5000, 5000, 21_000], dtype=np.uint64)
    src, dst = rng.integers(0, 300, 21_000, dtype=np.uint32), rng.integers(0, 300, 21_000, dtype=np.uint32)
    return offs, src, dst, *(torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst))


def _batch(ans, ctx, offs, src, dst, ds, dd, stream):
    out = torch.full((len(offs) - 1, 9), -1, dtype=torch.int64).pin_memory()
    _, summ, tk = ctx.batch_submit(ds, dd, offs, ans.BATCH_SUM, out=out, stream=stream)
    ctx.wait(tk)
    _, eq, esum = oracle.batch(src, dst, offs)
    assert ans.quantities_from_tensor(out) == eq
    assert summ.quantities() == oracle.network_quantities(esum)
    summ.free()


def test_batches_beside_other_contexts():
    from paper_2510_14050_gb300 import ans
    ans.load()
    mine, theirs = _data(1), _data(2)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    stop, errors = threading.Event(), []

    def run():
        try:
            while not stop.is_set():
                ctx = ans.Context(0)
                for path in (1, 0):  # (leaving path 1 waits for the device)
                    ctx.set_tuning(agg_path=path)
                    _batch(ans, ctx, *theirs, streams[1])
                ctx.set_wait_limit(0)
                ctx.close()
        except BaseException as e:
            errors.append(e)

    t = threading.Thread(target=run)
    t.start()
    ctx = ans.Context(0)
    try:
        end = time.perf_counter() + 2.0
        while time.perf_counter() < end and not errors:
            _batch(ans, ctx, *mine, streams[0])
    finally:
        stop.set()
        t.join()
    assert not errors, errors
    ctx.close()


FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef int (*end_fn)(void*, void**);
typedef int (*destroy_fn)(void*);
static int broken, seen;
void break_recordings(int n) { broken = n; }
int recordings(void) { return seen; }
int cudaStreamEndCapture(void* stream, void** graph) {
  void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  int e = ((end_fn)dlsym(rt, "cudaStreamEndCapture"))(stream, graph);
  ++seen;
  if (broken > 0 && e == 0) {
    --broken;
    ((destroy_fn)dlsym(rt, "cudaGraphDestroy"))(*graph);
    *graph = NULL;
    return 901; /* cudaErrorStreamCaptureInvalidated */
  }
  return e;
}
"""

CHILD = r"""
import ctypes, sys
import torch
sys.path.insert(0, "tests")
from test_gpu_threads import _batch, _data
from paper_2510_14050_gb300 import ans
fake = ctypes.CDLL(sys.argv[1])
data = _data(3)
for path in (0, 1):
    ctx = ans.Context(0)
    ctx.set_tuning(agg_path=path)
    for broken in (1, 0, 2, 0):
        fake.break_recordings(broken)
        n = fake.recordings()
        for _ in range(3):
            _batch(ans, ctx, *data, None)
        assert fake.recordings() == n + 3
    ctx.close()
print("CHILD OK")
"""


def test_a_recording_broken_off(tmp_path):
    (tmp_path / "fake.c").write_text(FAKE)
    lib = tmp_path / "fake.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(tmp_path / "fake.c"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=str(ROOT))
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "CHILD OK" in r.stdout, r.stdout + r.stderr
