"""The built-in force plans keep their partial sums within the room they are given (host code of
the library, no GPU)."""
import ctypes

import pytest

from paper_1409_5474_gb300 import build as nb_build


class Plan(ctypes.Structure):
    _fields_ = [(k, ctypes.c_int) for k in ("kind", "ipt", "threads", "nsplit", "jt", "nwj")]


@pytest.fixture(scope="module")
def lib():
    lib = ctypes.CDLL(nb_build.build())
    got = {}
    for order, plan, part in ((4, "_ZN2nb10plan_forceEiiiim", "_ZN2nb20plan_partial_doublesERKNS_9ForcePlanEi"),
                              (6, "_ZN2nb11plan_force6Eiiiim", "_ZN2nb21plan6_partial_doublesERKNS_9ForcePlanEi")):
        f, g = getattr(lib, plan), getattr(lib, part)
        f.restype, f.argtypes = Plan, [ctypes.c_int] * 4 + [ctypes.c_size_t]
        g.restype, g.argtypes = ctypes.c_size_t, [ctypes.POINTER(Plan), ctypes.c_int]
        got[order] = f, g
    return got


@pytest.mark.parametrize("order,variant", [(4, 0), (4, 1), (4, 2), (6, 1), (6, 2)])
@pytest.mark.parametrize("n_j", [1, 31, 300, 2500, 20011, 65536, 300000])
def test_partials_fit(lib, order, variant, n_j):
    plan, part = lib[order]
    for n_i in (1, 2, 4, 5, 8, 9, 31, 32, 33, 100, 512, 1531, 4095, 4096, 20000, 65536, 200000):
        free = plan(variant, n_i, n_j, 152, ctypes.c_size_t(-1).value)
        need = part(ctypes.byref(free), n_i)
        for room in (0, 1, 6, 7 * n_i, 20 * n_i, need // 2, max(need, 1) - 1, need, 2 * need):
            p = plan(variant, n_i, n_j, 152, room)
            assert p.nsplit >= 1
            assert part(ctypes.byref(p), n_i) <= room, (n_i, room, p.kind, p.nsplit)
            if room >= need:  # room enough: the plan is the free one
                assert [getattr(p, k) for k, _ in Plan._fields_] == \
                    [getattr(free, k) for k, _ in Plan._fields_]


# warp rows of the launch rule before the cost model, as a GB300 gave them
ROWS = {(2500, 300): 8, (8192, 380): 8, (8192, 498): 8, (20011, 300): 8, (20011, 498): 8,
        (65536, 300): 4, (65536, 498): 8, (131072, 498): 4}


@pytest.mark.parametrize("n_j,n_i", sorted(ROWS))
def test_order6_rows_of_257_to_511(lib, n_j, n_i):
    """More rows mean shorter FP32 sums: these sets keep the rows they had."""
    plan, _ = lib[6]
    assert plan(1, n_i, n_j, 152, ctypes.c_size_t(-1).value).nwj == ROWS[n_j, n_i]
