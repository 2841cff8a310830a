"""Routing (csrc/route.cuh, compiled here without CUDA): whatever the tables, classes, models, sizes and batch caps, every valid
placement goes to a kernel that its call launches.  A placement without one would keep its "not scored" record."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
OPTIMISTIC, FROZEN, MAXGAP, QUEUES = 1, 2, 4, 8
AUTO, BLOCK, GROUP, THREAD = 0, 1, 2, 3
MAX_ROWS = 256


@pytest.fixture(scope="module")
def routes(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("routes") / "libroutes.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-o", lib, os.path.join(HERE, "route_host.cpp")])
    lib = ctypes.CDLL(lib)
    u32, u64 = ctypes.c_uint32, ctypes.c_uint64
    lib.routes_unscored.restype = lib.routes_wide_from.restype = lib.routes_parts.restype = u32
    lib.routes_parts.argtypes = [u32, u64, u64]
    lib.routes_unscored.argtypes = [u32, u32, u64, u32, u32, u32, ctypes.POINTER(u32)]
    lib.routes_wide_from.argtypes = [u32, u32, u32, u32, u32, u64, u32, u32, u32]
    return lib


def _unscored(routes, flags, mapping, items, fits32=1, pool=0, hot=0):
    first = (ctypes.c_uint32 * 5)()
    n = routes.routes_unscored(flags, mapping, items, fits32, pool, hot, first)
    return n, dict(zip(("rows", "models", "classes", "instances", "cap"), first)) if n else None


@pytest.mark.parametrize("flags", [0, OPTIMISTIC, FROZEN, QUEUES])
@pytest.mark.parametrize("fits32", [1, 0])
@pytest.mark.parametrize("items", [1, 1000, 4096, 4097, 6000, 100_000, 10 ** 7])
def test_every_placement_has_a_kernel(routes, flags, fits32, items):
    assert _unscored(routes, flags, AUTO, items, fits32) == (0, None)


@pytest.mark.parametrize("mapping", [BLOCK, GROUP])
def test_every_placement_has_a_kernel_where_the_mapping_is_asked_for(routes, mapping):
    assert _unscored(routes, 0, mapping, 1000) == (0, None)
    assert _unscored(routes, MAXGAP, GROUP, 1000) == (0, None)


@pytest.mark.parametrize("pool, hot", [(128 << 10, 10 << 10), (30 << 10, 7 << 10), (4096, 1536), (8192, 2048)])
def test_every_placement_has_a_kernel_with_threads(routes, pool, hot):
    """(The pools' default sizes, and small ones that hold few instances.)"""
    assert _unscored(routes, 0, THREAD, 1000, 1, pool, hot) == (0, None)
    assert _unscored(routes, 0, AUTO, 1000, 1, pool, hot) == (0, None)


@pytest.mark.parametrize("flags", [0, OPTIMISTIC, FROZEN, QUEUES])
@pytest.mark.parametrize("items", [1000, 10 ** 6])
def test_large_tables_leave_the_walking_kernel_its_room(routes, flags, items):
    """The one-warp kernel, up to 592 MB of scratch, is launched for tables near the largest only, and there for placements near the
    largest: 16 models of 10 strategies are none of those."""
    for rows in range(1, MAX_ROWS + 1):
        for classes in (4, 71):
            first = routes.routes_wide_from(flags, AUTO, rows, 1, classes, items, 1, 0, 0)
            if rows <= 176 or flags in (FROZEN, QUEUES):
                assert first == 0, (rows, classes)
            else:
                assert first == 0 or first > 100, (rows, classes)
    assert routes.routes_wide_from(flags, AUTO, 160, 16, 71, items, 1, 0, 0) == 0


@pytest.mark.parametrize("models", [1, 2, 3, 8, 16])
@pytest.mark.parametrize("size", [1, 5, 17, 128])
def test_queues_are_replayed_in_parts_up_to_a_number_of_parts(routes, models, size):
    """Every part scans the whole trace: their number is bounded, however many models there are."""
    for items in (1, 100, 1000, 1330, 2000, 4000, 5328, 5329, 20_000):
        parts = routes.routes_parts(models, items, items * size)
        assert parts in (1, models)
        in_all = items * min(models, size)
        assert (parts == models) == (models == 1 or (items <= 3 * 148 * 12 and in_all <= 12 * 148 * 12)), (items, parts)
