"""Plan calls that run out of host memory (no GPU): the address space of a child
process ends at growing sizes, and every call returns AA_OK or AA_ERR_NOMEM; no
exception leaves the library, and a call that fails leaves the plan as it was."""
import subprocess
import sys

CHILD = r"""
import ctypes
import resource
import numpy as np
from paper_1912_07704_gb300 import abi
from paper_1912_07704_gb300.api import Plan

libc = ctypes.CDLL(None)
libc.mallopt(-3, 1 << 16)  # M_MMAP_THRESHOLD: what is freed leaves the address space
C, ndm = 1024, 300
make = lambda: Plan(C, 1508.0, -300.0 / C, 64e-6, [(0.0, 0.2, ndm, 1)])
N = 1 << 16
def least(p): return abi.aa_dedisperse_least_ws_bytes(p.handle, N)
with make() as p:  # code and first-use data are in place
    want = abi.aa_plan_effective_shifts(p.handle, 0, ndm, C)
    assert p.query(N).dedisp_ws_bytes > least(p)
    p.set_fdmt(0)
    tree = abi.aa_plan_effective_shifts(p.handle, 0, ndm, C)
out = np.zeros((ndm, C), np.int32)
def shifts(p):  # (into memory that is there)
    abi.check(abi.lib().aa_plan_effective_shifts(p.handle, 0, out.ctypes.data, out.size), "shifts")
    return out
hard = resource.getrlimit(resource.RLIMIT_AS)[1]
seen = {"plan": set(), "without bands": set(), "tree": set(), "shifts": set()}
def size():
    return int(open("/proc/self/statm").read().split()[0]) * 4096
def limited(quarter_mb, fn):
    libc.malloc_trim(0)
    resource.setrlimit(resource.RLIMIT_AS, (size() + quarter_mb * (1 << 18), hard))
    try:
        return fn()
    except abi.AAError as e:
        assert e.status == abi.AA_ERR_NOMEM, e
        return None
    except MemoryError:  # (the interpreter's own)
        return None
    finally:
        resource.setrlimit(resource.RLIMIT_AS, (hard, hard))
for quarter_mb in list(range(0, 80)) + [120, 200, 400, 2000]:
    p = limited(quarter_mb, make)
    seen["plan"].add(p is not None)
    if p is not None:
        seen["without bands"].add(p.query(N).dedisp_ws_bytes == least(p))
        assert np.array_equal(abi.aa_plan_effective_shifts(p.handle, 0, ndm, C), want)
        p.close()
for quarter_mb in range(0, 24):
    with make() as p:
        done = limited(quarter_mb, lambda: p.set_fdmt(0) or True)
        seen["tree"].add(done is not None)
        assert np.array_equal(abi.aa_plan_effective_shifts(p.handle, 0, ndm, C), tree if done else want)
    with make() as p:
        got = limited(quarter_mb, lambda: shifts(p))
        assert got is None or np.array_equal(got, want)
        p.set_fdmt(0)
        got = limited(quarter_mb, lambda: shifts(p))
        seen["shifts"].add(got is not None)
        assert got is None or np.array_equal(got, tree)
assert all(v == {True, False} for v in seen.values()), seen
print("ok", seen)
"""


def test_no_exception_leaves_the_library():
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout[-500:], r.stderr[-2000:])
