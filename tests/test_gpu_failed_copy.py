"""A batch whose copy of the quantities to pageable host memory fails (the
runtime's answer is a fake's, in a child process) gives its blocks back and
leaves the context usable."""
import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

ROOT = Path(__file__).resolve().parent.parent

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef int (*copy_fn)(void*, const void*, size_t, int, void*);
static void* refuse;
void refuse_copy_to(void* dst) { refuse = dst; }
int cudaMemcpyAsync(void* dst, const void* src, size_t n, int kind, void* stream) {
  static copy_fn real;
  if (refuse && dst == refuse) {
    refuse = NULL;
    return 1; /* cudaErrorInvalidValue */
  }
  if (!real) real = (copy_fn)dlsym(dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD), "cudaMemcpyAsync");
  return real(dst, src, n, kind, stream);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np, torch
import oracle
from paper_2510_14050_gb300 import ans
fake = ctypes.CDLL(sys.argv[1])
rng = np.random.default_rng(1)
offs = np.array([0, 20000, 30001], dtype=np.uint64)
src, dst = rng.integers(0, 99, 30001, dtype=np.uint32), rng.integers(0, 99, 30001, dtype=np.uint32)
ds, dd = (torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst))
_, eq, esum = oracle.batch(src, dst, offs)
ctx = ans.Context(0)
out = torch.zeros((2, 9), dtype=torch.int64)
def batch():
    mats, summ, tk = ctx.batch_submit(ds, dd, offs, ans.BATCH_MATRICES | ans.BATCH_SUM, out=out)
    ctx.wait(tk)
    assert ans.quantities_from_tensor(out) == eq
    assert all(np.array_equal(a, b) for a, b in zip(summ.to_numpy(), esum))
    for m in [*mats, summ]:
        m.free()
batch()
held = ctx.memory()[0]
fake.refuse_copy_to(ctypes.c_void_p(out.data_ptr()))
try:
    batch()
    raise SystemExit("the copy was not refused")
except ans.AnsError as e:
    assert e.code == ans.ERR_CUDA, e
assert ctx.memory()[0] == held, (ctx.memory()[0], held)
batch()
assert ctx.memory()[0] == held
ctx.close()
print("CHILD OK")
"""


def test_blocks_are_given_back(tmp_path):
    (tmp_path / "fake.c").write_text(FAKE)
    lib = tmp_path / "fake.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(tmp_path / "fake.c"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=str(ROOT))
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "CHILD OK" in r.stdout, r.stdout + r.stderr
