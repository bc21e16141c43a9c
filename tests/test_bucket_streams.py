"""How rr_bucket_route_layer orders its buckets, on the host: the bucket front end compiled against a
stand-in for streams, events and ledger calls (fake_streams.cpp) that records what is ordered before
what.  No GPU."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200.build import CSRC, _nvcc

HERE = os.path.dirname(os.path.abspath(__file__))
MAIN = 1000                                     # the caller's stream
WIDTHS = [8, 16, 32, 8, 16, 32]                 # (a stand-in ledger is named by its width)


@pytest.fixture(scope="module")
def lib_path(tmp_path_factory):
    d = tmp_path_factory.mktemp("buckets")
    objs = []
    for src in (os.path.join(CSRC, "rr_buckets.cu"), os.path.join(HERE, "fake_streams.cpp")):
        obj = str(d / (os.path.basename(src) + ".o"))
        subprocess.run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-Xcompiler", "-fPIC",
                        "-c", src, "-o", obj], check=True)
        objs.append(obj)
    out = str(d / "libbuckets.so")
    subprocess.run([shutil.which("g++") or "g++", "-shared", "-Wl,-Bsymbolic", "-o", out] + objs, check=True)
    return out


@pytest.fixture
def side(lib_path, tmp_path):
    """A fresh copy of the library (its own record) and a set of three buckets."""
    own = str(tmp_path / "libbuckets.so")
    shutil.copy(lib_path, own)
    lib = C.CDLL(own, mode=os.RTLD_LOCAL | os.RTLD_NOW)
    cfg = B.rr_config(batch=1, heads=len(WIDTHS), n_q=64, n_k=64, d=64, k=8, dtype=B.RR_BF16)
    handle = C.c_void_p()
    w = (C.c_int32 * len(WIDTHS))(*WIDTHS)
    assert lib.rr_bucket_set_init(C.byref(cfg), w, len(WIDTHS), C.c_void_p(1 << 20), C.c_size_t(1 << 16),
                                  C.c_void_p(1 << 21), C.c_size_t(1 << 16), C.byref(handle)) == B.RR_OK
    yield lib, lambda layer, anchor=0: lib.rr_bucket_route_layer(handle, C.c_void_p(4096), C.c_void_p(8192), layer,
                                                                 anchor, C.c_void_p(MAIN))
    lib.rr_bucket_set_destroy(handle)


def test_buckets_are_unordered_among_themselves_and_ordered_on_the_callers_stream(side):
    lib, route = side
    before = lib.fake_op(C.c_void_p(MAIN))
    last = [before]
    for layer in range(3):
        first = lib.fake_count()
        assert route(layer, 1 if layer == 0 else 0) == B.RR_OK
        ops = list(range(first, lib.fake_count()))
        assert sorted(lib.fake_ledger(o) for o in ops) == [8, 16, 32]
        for o in ops:                            # behind everything the caller enqueued, and the layer before
            assert all(lib.fake_before(p, o) for p in last)
        for a in ops:                            # side by side, the narrowest bucket included
            assert not any(lib.fake_before(a, b) for b in ops if b != a), lib.fake_ledger(a)
        after = lib.fake_op(C.c_void_p(MAIN))
        assert all(lib.fake_before(o, after) for o in ops)
        last = ops + [after]


@pytest.mark.parametrize("failing", [8, 16, 32])
def test_a_failed_bucket_leaves_what_was_enqueued_ordered(side, failing):
    lib, route = side
    lib.fake_fail(failing, 0)
    first = lib.fake_count()
    assert route(0, 1) == B.RR_ERR_UNSUPPORTED
    ops = list(range(first, lib.fake_count()))
    assert len(ops) == {32: 0, 16: 1, 8: 2}[failing]
    after = lib.fake_op(C.c_void_p(MAIN))
    assert all(lib.fake_before(o, after) for o in ops)


def test_a_failed_fork_is_reported_and_the_others_are_joined(side):
    lib, route = side
    lib.fake_fail(0, 2)                          # the second bucket's wait for the caller's stream
    first = lib.fake_count()
    assert route(0, 1) == B.RR_ERR_CUDA
    ops = list(range(first, lib.fake_count()))
    assert [lib.fake_ledger(o) for o in ops] == [32]
    after = lib.fake_op(C.c_void_p(MAIN))
    assert lib.fake_before(ops[0], after)
