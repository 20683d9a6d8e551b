"""Contexts in less than the workspace of the fastest form: fewer chunks and instances at a time, FP64 units."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _least(d, dcut, batch, kw):
    from paper_1906_06060_gb300 import _lib, _opts
    o = _opts(kw["precision"], batch, kw.get("fp64_steps", 2), 64, derivatives=kw.get("derivatives", False),
              impurities=kw.get("impurities", False), z2=kw.get("z2", False))
    n, least = ctypes.c_size_t(), ctypes.c_size_t()
    _lib.load().hotrg_workspace_size(d, dcut, ctypes.byref(o), ctypes.byref(n))
    _lib.load().hotrg_workspace_min(d, dcut, ctypes.byref(o), ctypes.byref(least))
    return n.value, least.value


CASES = [(4, [0.1497], 5, 6, dict(precision="fp64")), (4, [0.14, 0.1497, 0.16], 5, 5, dict(precision="fp64")),
         (4, [0.1497], 5, 5, dict(precision="fp64", z2=True)),
         (4, [0.1497, 0.15], 5, 4, dict(precision="fp64", derivatives="eig")),
         (4, [0.1497, 0.15], 5, 4, dict(precision="fp64", impurities=True)),
         (3, [0.22], 10, 5, dict(precision="fp64")), (2, [0.44] * 5, 8, 8, dict(precision="fp64")),
         (4, [0.14, 0.1497, 0.16], 5, 6, dict(precision="fp16x3", fp64_steps=3))]


@pytest.mark.parametrize("d,beta,dcut,steps,kw", CASES)
def test_smaller_workspaces_give_the_same_flow(d, beta, dcut, steps, kw):
    """From the full size down to the least, halving: FP64 rounding in every form of an FP64 context (1e-12; the products
    may run on the FP64 units, the Gram sums in fewer splits), the split's own accuracy in a split one (1e-7). Less than the
    least is refused."""
    from paper_1906_06060_gb300 import HOTRG, HotrgError, _lib
    n, least = _least(d, dcut, len(beta), kw)
    h = 0.0 if kw.get("z2") else 0.01
    keys = ("lnz_per_site", "dlnz_dbeta", "dlnz_dh", "nn_correlation", "spin")
    ref = None
    while True:
        with HOTRG(d, beta, h, dcut, workspace=n, **kw) as f:
            for _ in range(steps):
                f.step()
            obs = [f.observables(i) for i in range(len(beta))]
        got = np.array([[o[k] for k in keys] for o in obs])
        ref = got if ref is None else ref
        np.testing.assert_allclose(got, ref, rtol=1e-12 if kw["precision"] == "fp64" else 1e-7, atol=1e-13)
        if n == least:
            break
        n = max(n // 2, least)
    with pytest.raises(HotrgError) as e:
        HOTRG(d, beta, h, dcut, workspace=least - 256, **kw)
    assert e.value.code == _lib.HOTRG_ENOMEM


def test_a_full_device_gets_a_smaller_workspace(monkeypatch):
    """The binding halves the workspace where the device does not have the full one free, and gives up below the least."""
    import torch
    from paper_1906_06060_gb300 import HOTRG
    n, least = _least(4, 5, 1, dict(precision="fp64"))
    free, empty = n // 5, torch.empty

    def limited(size, **kw):
        if size > free:
            raise torch.cuda.OutOfMemoryError("limited")
        return empty(size, **kw)

    with HOTRG(4, 0.1497, 0.01, 5) as f:
        for _ in range(4):
            f.step()
        ref = f.free_energy()[0]
    monkeypatch.setattr(torch, "empty", limited)
    with HOTRG(4, 0.1497, 0.01, 5) as f:
        assert least <= f._ws.numel() <= free
        for _ in range(4):
            f.step()
        np.testing.assert_allclose(f.free_energy()[0], ref, rtol=1e-13)
    free = least - 1
    with pytest.raises(torch.cuda.OutOfMemoryError):
        HOTRG(4, 0.1497, 0.01, 5)
