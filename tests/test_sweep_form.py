"""The form of the warp-strip sweep (operand ring, edge buffers) that a level takes where the device holds a
cluster of more than eight CTAs only with little shared memory: the form is one that can be launched, not one
that a smaller relative of it can, and without any the level takes another sweep.  Host only."""
import ctypes

import pytest

LIMIT = 227 * 1024


def _form(ni, nj, nw, deep=1, cluster_bytes=LIMIT):
    import paper_1710_04875_gb300 as P
    stages, edges, nbytes = ctypes.c_int(), ctypes.c_int(), ctypes.c_longlong()
    assert P.library().fasw_check_sweep_form(ni, nj, nw, deep, cluster_bytes, ctypes.byref(stages),
                                             ctypes.byref(edges), ctypes.byref(nbytes)) == 0
    return stages.value, edges.value, nbytes.value


@pytest.mark.parametrize("ni,nj,nw", [(1024, 256, 128), (64, 250, 8), (300, 129, 30), (1024, 129, 128)])
def test_the_form_taken_is_one_the_device_holds(ni, nj, nw):
    full, shallow = _form(ni, nj, nw), _form(ni, nj, nw, deep=0)
    assert full[:2] == (5, 2) and shallow[:2] == (3, 2) and shallow[2] < full[2] <= LIMIT
    seen = []
    for cluster_bytes in range(full[2], 0, -1024):
        for deep in (1, 0):
            form = _form(ni, nj, nw, deep, cluster_bytes)
            assert form[2] <= cluster_bytes and (deep or form[0] in (0, 3))
            seen.append(form[:2])
    assert {(5, 2), (3, 2), (3, 1), (0, 0)} <= set(seen)


@pytest.mark.parametrize("ni,nj,nw,form", [(1024, 128, 128, (5, 2)), (10, 2, 2, (5, 2)), (4200, 10, 0, (3, 1)),
                                           (6000, 10, 0, (0, 0)), (64, 257, 8, (0, 0))])
def test_portable_clusters_ask_for_shared_memory_alone(ni, nj, nw, form):
    assert _form(ni, nj, nw, cluster_bytes=1)[:2] == form


def test_bad_arguments():
    import paper_1710_04875_gb300 as P
    lib, n, b = P.library(), ctypes.c_int(), ctypes.c_longlong()
    assert lib.fasw_check_sweep_form(0, 8, 0, 1, 0, ctypes.byref(n), ctypes.byref(n), ctypes.byref(b)) == -1
    assert lib.fasw_check_sweep_form(64, 8, 0, 1, -1, ctypes.byref(n), ctypes.byref(n), ctypes.byref(b)) == -1
    assert lib.fasw_check_sweep_form(64, 8, 0, 1, 0, None, ctypes.byref(n), ctypes.byref(b)) == -1
