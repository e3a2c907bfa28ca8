"""The C-ABI library loads and exports every function include/retexo.h
declares; host-side argument validation rejects bad calls before any launch
(no GPU needed: these calls return before touching the device)."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "include", "retexo.h")


@pytest.fixture(scope="module")
def lib():
    from paper_2302_13053_b200 import build
    return C.CDLL(build.build())


def declared_functions():
    text = open(HEADER).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(retexo_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_function_is_exported(lib):
    names = declared_functions()
    assert {"retexo_aggregate", "retexo_mlp_train_step", "retexo_embed", "retexo_cross_partition_bytes",
            "retexo_lmp_train"} <= set(names)
    for name in names:
        assert hasattr(lib, name), name
    from paper_2302_13053_b200 import binding
    assert sorted(binding.EXPORTS) == names


def test_status_strings_and_sizes(lib):
    lib.retexo_status_string.restype = C.c_char_p
    assert lib.retexo_status_string(0) == b"ok"
    assert len({lib.retexo_status_string(i) for i in range(8)}) == 8
    lib.retexo_theta_size.restype = C.c_int64
    assert lib.retexo_theta_size(C.c_int32(10), C.c_int32(4), C.c_int32(3)) == 10 * 4 + 4 + 4 * 3 + 3
    assert lib.retexo_theta_size(C.c_int32(10), C.c_int32(0), C.c_int32(3)) == 33
    for fn in ("retexo_aggregate_workspace_size", "retexo_cross_partition_workspace_size"):
        getattr(lib, fn).restype = C.c_size_t
    assert lib.retexo_aggregate_workspace_size(C.c_int64(1000), C.c_int64(5000), C.c_int32(0), C.c_int32(64),
                                               C.c_int32(0)) >= 1000 * 4
    small = lib.retexo_cross_partition_workspace_size(C.c_int64(1000), C.c_int64(5000), C.c_int32(100))
    big = lib.retexo_cross_partition_workspace_size(C.c_int64(1000), C.c_int64(5000), C.c_int32(1000000))
    assert 0 < small < big


def test_aggregation_workspace_holds_a_copy_of_the_rows_only_where_one_is_made(lib):
    lib.retexo_aggregate_workspace_size.restype = C.c_size_t

    def size(n, e, dim, type=0):
        return lib.retexo_aggregate_workspace_size(C.c_int64(n), C.c_int64(e), C.c_int32(type), C.c_int32(dim), C.c_int32(0))

    partial = size(2449029, 123718280, 100, type=1)                     # mean: segment sums alone
    assert partial < 250 << 20
    # the rows stay where they are: bound by memory, or copies beyond 2 GB
    for n, e, dim in ((2449029, 123718280, 100), (2449029, 123718280, 256), (4000000, 4000000, 512)):
        assert size(n, e, dim) - size(n, e, dim, type=1) < 4 * n + 1024
    assert 4 * 100000 * 100 <= size(100000, 4000000, 100) - size(100000, 4000000, 100, type=1) <= 4 * 100000 * 132   # scaled rows


def test_host_features_need_no_second_matrix_on_the_device(lib):
    from paper_2302_13053_b200.binding import _LmpConfig
    lib.retexo_lmp_workspace_size.restype = C.c_size_t
    n, e = 2449029, 123718280

    def size(d0, host):
        cfg = _LmpConfig(0, 2, 10, d0, 64, 47, 0, 0.01, 0.9, 0.999, 1e-8, 1, 0, 0, 0.2, host, 0.0, 0, 0, 0, 1e-5, 0.1)
        return lib.retexo_lmp_workspace_size(C.byref(cfg), C.c_int64(n), C.c_int64(e), C.c_int64(200000), C.c_int64(40000),
                                             C.c_int64(2000000), C.c_int32(0))

    # rows of 99 columns are re-laid on the device from pieces of 64 MB; rows of 100 stay as they come
    assert size(100, 0) > 0
    assert 0 < size(99, 1) - size(100, 1) <= (64 << 20)


def test_standard_training_holds_no_copy_of_the_features(lib):
    from paper_2302_13053_b200.binding import _StandardConfig
    lib.retexo_standard_workspace_size.restype = C.c_size_t
    n = 232965

    def size(d0):
        cfg = _StandardConfig(1, 2, 10, d0, 256, 41, 0, 0.01, 0.9, 0.999, 1e-8)
        return lib.retexo_standard_workspace_size(C.byref(cfg), C.c_int64(n), C.c_int64(1000000), C.c_int64(100000), C.c_int64(10000),
                                                  C.c_int64(20000))

    # [X^1 | 1] has 1216 columns of 2 bytes either way; rows of 608 columns instead of 576 are 30 MB of a copy (parameters: 5 MB)
    assert 0 < size(576) <= size(607) < size(576) + (16 << 20)


def test_bad_arguments_are_rejected_on_the_host(lib):
    from paper_2302_13053_b200.binding import _Csr, _Mlp
    INVALID, WORKSPACE = 1, 4
    g = _Csr(-1, 0, None, None)
    assert lib.retexo_aggregate(C.byref(g), 0, None, C.c_int64(4), 4, None, None, C.c_int64(4), 1, None,
                                C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    g = _Csr(0, 0, None, None)       # an empty graph is a valid no-op
    assert lib.retexo_aggregate(C.byref(g), 0, None, C.c_int64(4), 4, None, None, C.c_int64(4), 1, None,
                                C.c_int64(0), None, C.c_size_t(0), None) == 0
    g = _Csr(4, 0, 1, None)          # null feature pointer, no outputs
    assert lib.retexo_aggregate(C.byref(g), 0, None, C.c_int64(4), 4, None, None, C.c_int64(4), 1, None,
                                C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    assert lib.retexo_aggregate(C.byref(g), 7, C.c_void_p(256), C.c_int64(4), 4, None, C.c_void_p(256),
                                C.c_int64(4), 1, None, C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    # valid shapes but no workspace
    assert lib.retexo_aggregate(C.byref(g), 0, C.c_void_p(256), C.c_int64(4), 4, None, C.c_void_p(256),
                                C.c_int64(4), 1, None, C.c_int64(0), None, C.c_size_t(0), None) == WORKSPACE
    dims = (C.c_int32 * 1)(4)
    assert lib.retexo_cross_partition_bytes(C.byref(g), C.c_void_p(256), 0, 1, dims, 4, None, None, None, None,
                                            None, None, None, C.c_size_t(0), None) == INVALID
    m = _Mlp(0, 4, 3, 256, None, None, 1, 0.1, 0.9, 0.999, 1e-8, 0)
    assert lib.retexo_mlp_train_step(C.byref(m), C.c_void_p(256), C.c_int64(8), C.c_int32(0),
                                     C.c_void_p(256), C.c_int64(4), None, None, None, C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    m = _Mlp(8, 4, 3, 256, None, None, 1, 0.1, 0.9, 0.999, 1e-8, 0)      # Adam without moments
    assert lib.retexo_mlp_train_step(C.byref(m), C.c_void_p(256), C.c_int64(8), C.c_int32(0),
                                     C.c_void_p(256), C.c_int64(4), None, None, None, C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    m = _Mlp(8, 4, 3, 256, None, None, 0, 0.1, 0.9, 0.999, 1e-8, 0)
    ALIGNMENT = 3
    assert lib.retexo_mlp_train_step(C.byref(m), C.c_void_p(256), C.c_int64(9), C.c_int32(0),
                                     C.c_void_p(256), C.c_int64(4), None, None, None, C.c_int64(0), None, C.c_size_t(0), None) == ALIGNMENT
    # a column of ones is claimed, but the rows have no room for it
    assert lib.retexo_mlp_train_step(C.byref(m), C.c_void_p(256), C.c_int64(8), C.c_int32(1),
                                     C.c_void_p(256), C.c_int64(4), None, None, None, C.c_int64(0), None, C.c_size_t(0), None) == INVALID
    assert lib.retexo_embed(C.byref(m), C.c_void_p(256), C.c_int64(8), None, C.c_int64(4), None, C.c_int64(0), None,
                            C.c_int64(0), None, C.c_int64(0), None, None, None, None, C.c_size_t(0), None) == WORKSPACE
