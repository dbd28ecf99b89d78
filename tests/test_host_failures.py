"""What a handle does after a CUDA call has failed on the host: the library's
host code, linked with a fake runtime whose n-th call of a kind fails, so no
GPU is needed and none is disturbed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2205_11048_gb300 import binding as B
from paper_2205_11048_gb300 import build as BLD

HERE = os.path.dirname(os.path.abspath(__file__))
MALLOC, MEMCPY_ASYNC, PUSH_COPY = 0, 1, 2


@pytest.fixture(scope="module")
def F(tmp_path_factory):
    BLD.build()
    out = tmp_path_factory.mktemp("fake")
    objs, lib = [os.path.join(BLD.OUT_DIR, "gba_host.o")], str(out / "libgba_fake.so")
    cc = [BLD.nvcc(), *BLD.ARCH]
    for src in ("fake_runtime.cpp", "fake_launchers.cu"):
        objs.append(str(out / (src + ".o")))
        subprocess.run([*cc, *BLD.FLAGS, "-I" + BLD.CSRC, "-c", os.path.join(HERE, src), "-o", objs[-1]],
                       check=True)
    subprocess.run([*cc, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", lib, *objs], check=True)
    L = ctypes.CDLL(lib)
    for name, (res, args) in B._SIGNATURES.items():
        if hasattr(L, name):
            getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.fake_allocations.restype = ctypes.c_long
    return L


@pytest.fixture(autouse=True)
def _clean(F):
    F.fake_addressable(0)
    for kind in (MALLOC, MEMCPY_ASYNC, PUSH_COPY):
        F.fake_fail(kind, 0)
    F.cudaGetLastError()
    n, bad = F.fake_allocations(), F.fake_bad()
    yield
    while Handle.open:
        F.gba_destroy(Handle.open.pop())
    assert F.fake_bad() == bad, "a launcher was given memory that is not there"
    assert F.fake_allocations() == n, "allocations outlive their handle"


class Handle:
    open = []

    def __init__(self, F, dim=4, mode=0, G=3, max_buf=3, max_ids=8, D=8, rows=100, kind=0, more=None):
        self.F, self.dim, self.D = F, dim, D
        self.h = ctypes.c_void_p()
        tables = [B.gba_table_desc(rows, dim, mode, max_ids, B.opt_desc(kind, 0.01))] + (more or [])
        self.T = len(tables)
        assert F.gba_create((B.gba_table_desc * self.T)(*tables), self.T, D, ctypes.byref(B.opt_desc()), G, max_buf, None,
                            0, None, ctypes.byref(self.h)) == B.GBA_OK
        Handle.open.append(self.h)
        self.keep = []

    def push(self, n=5, ref=False):
        ids, rows, dense = np.arange(n), np.zeros((n, self.dim), np.float32), np.zeros(self.D + 4, np.float32)
        at = (dense.ctypes.data + 15) & ~15
        self.keep.append((ids, rows, dense))
        g = (B.gba_sparse_grad * self.T)(*[B.gba_sparse_grad(ids.ctypes.data, n, rows.ctypes.data)] * self.T)
        return (self.F.gba_push_ref if ref else self.F.gba_push)(self.h, 0, g, at, 1)

    def apply(self):
        return self.F.gba_try_apply(self.h)

    def arrays(self):
        p = [ctypes.c_void_p() for _ in range(4)]
        assert self.F.gba_get_table(self.h, 0, *[ctypes.byref(x) for x in p]) == B.GBA_OK
        return [x.value for x in p]

    def capacity(self):
        n = ctypes.c_int64()
        assert self.F.gba_table_capacity(self.h, 0, ctypes.byref(n)) == B.GBA_OK
        return n.value


@pytest.mark.parametrize("eager", [False, True])
@pytest.mark.parametrize("kind,nth", [(PUSH_COPY, 1), (MEMCPY_ASYNC, 1), (MEMCPY_ASYNC, 2), (MEMCPY_ASYNC, 3)])
def test_a_push_whose_copy_failed_takes_no_place_in_the_buffer(F, kind, nth, eager):
    """A copying push that returns an error stores no message, so it holds no
    dense slot and no space for ids either, and its error is not reported a
    second time by the step that follows."""
    h = Handle(F)
    if eager:
        assert F.gba_set_eager_dense(h.h, 1) == B.GBA_OK
    F.fake_addressable(kind == PUSH_COPY)
    assert h.push() == B.GBA_OK
    for _ in range(10):
        F.fake_fail(kind, nth)
        assert h.push() == B.GBA_E_CUDA
        assert F.gba_last_error(h.h)
    assert [h.push() for _ in range(3)] == [B.GBA_OK, B.GBA_OK, B.GBA_E_FULL]
    assert h.apply() == 1 and h.apply() == 0
    assert [h.push() for _ in range(4)] == [B.GBA_OK] * 3 + [B.GBA_E_FULL]
    assert h.apply() == 1


@pytest.mark.parametrize("n,nth", [(100_000, 1)] + [(10_000, n) for n in range(1, 21)])
def test_a_step_whose_buffers_could_not_grow_is_refused_until_they_can(F, n, nth):
    """The n-th allocation of the step's buffers fails: the step is not applied
    and stays buffered, a smaller one does not run on what is left of the
    buffers, and the next that finds memory allocates them."""
    h = Handle(F, G=1, max_buf=4, max_ids=200_000, dim=20)
    assert h.push(n=600, ref=True) == B.GBA_OK
    assert h.apply() == 1
    assert h.push(n=n, ref=True) == B.GBA_OK and h.push(n=10, ref=True) == B.GBA_OK
    for _ in range(2):
        F.fake_fail(MALLOC, nth)
        assert h.apply() == B.GBA_E_OOM
    assert F.gba_pull_version(h.h) == 1
    n_sorted = ctypes.c_int64()  # the record of the step before went with its buffers
    assert F.gba_debug_sorted(h.h, 0, None, None, ctypes.byref(n_sorted)) == B.GBA_E_STATE
    assert [h.apply(), h.apply(), h.apply()] == [1, 1, 0]


# four arrays, five with Adam's second moment
@pytest.mark.parametrize("kind,nth", [(0, n) for n in range(1, 5)] + [(1, n) for n in range(1, 6)])
def test_a_hash_table_that_could_not_grow_keeps_its_rows(F, kind, nth):
    """The n-th of the larger table's allocations fails: the step is refused,
    the table stays as it is, and a later step grows it."""
    h = Handle(F, G=1, max_buf=4, max_ids=4096, rows=1024, mode=B.HASH, kind=kind)
    assert h.push(n=400, ref=True) == B.GBA_OK
    assert h.apply() == 1
    before, n = h.arrays(), F.fake_allocations()
    assert h.push(n=600, ref=True) == B.GBA_OK
    for _ in range(2):
        F.fake_fail(MALLOC, nth)
        assert h.apply() == B.GBA_E_OOM
        assert (h.arrays(), h.capacity(), F.fake_allocations()) == (before, 1024, n)
    assert h.apply() == 1
    assert h.capacity() == 2048


@pytest.mark.parametrize("nth", range(5, 9))
def test_the_second_of_two_hash_tables_could_not_grow(F, nth):
    """The first table has grown when the second cannot: the steps that follow
    find the first where it is now."""
    h = Handle(F, G=1, max_buf=4, max_ids=4096, rows=1024, mode=B.HASH,
               more=[B.gba_table_desc(1024, 4, B.HASH, 4096, B.opt_desc(0, 0.01))])
    assert h.push(n=600, ref=True) == B.GBA_OK
    F.fake_fail(MALLOC, nth)
    assert h.apply() == B.GBA_E_OOM
    assert h.capacity() == 2048
    assert h.apply() == 1


def test_a_hash_table_does_not_grow_past_the_keys(F):
    """Growth that would bring the tables to 2^32 - 1 rows is refused before
    anything changes: the table keeps its rows, and the handle is not failed."""
    h = Handle(F, G=1, max_buf=4, max_ids=4096, rows=1024, mode=B.HASH, dim=1,
               more=[B.gba_table_desc(2**32 - 2 - 1024, 1, B.DIRECT, 4096, B.opt_desc(0, 0.01))])
    assert h.push(n=600, ref=True) == B.GBA_OK
    before = h.arrays()
    for _ in range(3):
        assert h.apply() == B.GBA_E_ARG
    assert (h.arrays(), h.capacity()) == (before, 1024)
    assert F.gba_sync(h.h) == B.GBA_OK


def test_fresh_buffers_are_filled_in_the_order_of_the_handles_streams(F):
    """Nothing clears or fills device memory on the default stream: the first
    copies of a push and the first kernels of a step do not wait for it, so a
    clear still under way would take what they have written (a race, so it is
    shown here and not on a GPU)."""
    before = F.fake_unordered()
    h = Handle(F, G=1, max_buf=4, max_ids=4096, rows=1024, mode=B.HASH)
    assert [h.push(n=600), h.apply(), h.push(n=4000), h.apply()] == [B.GBA_OK, 1, B.GBA_OK, 1]
    assert h.capacity() > 1024
    assert F.fake_unordered() == before
