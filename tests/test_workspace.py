"""Workspace plans: the size of the fastest form of the steps, and the least that holds a context."""
import ctypes

import pytest

MB = 10 ** 6


@pytest.fixture(scope="module")
def sizes():
    from paper_1906_06060_gb300 import _lib, _opts, build
    build.build()
    lib = _lib.load()

    def get(d, dcut, precision, batch=1, **kw):
        o = _opts(precision, batch, 2, 64, **kw)
        n, least = ctypes.c_size_t(), ctypes.c_size_t()
        assert lib.hotrg_workspace_size(d, dcut, ctypes.byref(o), ctypes.byref(n)) == 0
        assert lib.hotrg_workspace_min(d, dcut, ctypes.byref(o), ctypes.byref(least)) == 0
        return n.value, least.value
    return get


# bytes in which each context fits with one chunk of a squeeze in flight and FP64 operands
@pytest.mark.parametrize("d,dcut,precision,kw,holds", [
    (2, 8, "fp64", {}, 41.7 * MB), (2, 16, "fp64", {}, 109.5 * MB), (3, 10, "fp64", {}, 281.9 * MB),
    (4, 4, "fp64", {}, 11.8 * MB), (4, 5, "fp64", {"batch": 16}, 491.6 * MB), (4, 5, "fp64", {"z2": True}, 62.9 * MB),
    (4, 5, "fp64", {"derivatives": "eig"}, 149.8 * MB), (4, 6, "fp16x3", {"impurities": True}, 213.4 * MB),
    (4, 8, "bf16x6", {}, 2043.2 * MB), (4, 10, "fp64", {"batch": 16}, 180713 * MB), (4, 13, "bf16x6", {}, 137633 * MB)])
def test_least_workspace_needs_no_batches_and_no_digits(sizes, d, dcut, precision, kw, holds):
    n, least = sizes(d, dcut, precision, **kw)
    assert least <= holds and least <= n


def test_fp64_contexts_give_up_instances_before_digits(sizes):
    """16 instances at bond dimension 10: groups of eight with digit planes pass 128 GiB, smaller groups do not. The
    FP64 operands of a group of eight alone take 180 GB."""
    n, _ = sizes(4, 10, "fp64", batch=16)
    assert n <= 128 << 30


def test_arguments_are_checked():
    from paper_1906_06060_gb300 import _lib, build
    build.build()
    lib = _lib.load()
    n = ctypes.c_size_t()
    for bad in [(0, 4), (5, 4), (4, 1), (4, 17)]:
        assert lib.hotrg_workspace_min(bad[0], bad[1], None, ctypes.byref(n)) == _lib.HOTRG_EINVAL
    assert lib.hotrg_workspace_min(4, 4, None, None) == _lib.HOTRG_EINVAL
