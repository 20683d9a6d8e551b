"""Performance cases of the HOTRG library: what its users have it do, through its public entry points.

Five kinds of call:
  flow    a whole coarse-graining flow of the Ising model: a context, n steps, ln Z/N read back after every
          step (2D, 3D and 4D; one temperature or a temperature / field scan in one context)
  grad    ln Z/N and its derivatives in (beta, h) through torch.autograd
  step    one coarse-graining step of a checkpointed tensor: restore, step, read ln Z/N and the tensor
  steady  the next step of a running flow at the paper's scale (4D, bond dimension 10)
  gemm    the split-precision GEMM on its own

Results of FP64 calls are returned in 64 bits. Results of the split-precision modes (bf16x3/x4/x6, fp16x3/x4)
are returned in 32 bits, the precision in which those modes hold their intermediates (their specified accuracy
is 1e-7 on ln Z/N). The tensors of an Ising flow are unique only up to rotations inside exactly degenerate
multiplets of their Gram spectra, so the flows return their gauge-invariant results; the steps start from tensors
with generic spectra and return the whole new tensor.
"""
import itertools
import math

import numpy as np
import torch

from paper_1906_06060_gb300 import HOTRG, gemm_split
from paper_1906_06060_gb300.autograd import lnz as lnz_autograd

# Bond dimensions at which no cut of the zero-field Ising flows splits a degenerate multiplet (at the others the
# truncated flow itself is not unique).
CLEAN_DCUT = {2: (4, 5, 6, 8, 10, 12), 3: (4, 5, 6, 10), 4: (3, 5)}
BETA = {2: (0.30, 0.44), 3: (0.20, 0.24), 4: (0.14, 0.16)}


def listed():
    return [
        # the smallest whole call: a 2D flow to 1024^2 (the 2D check of the method), every step launch- and
        # latency-bound
        {"name": "flow_2d_d8", "kind": "flow", "d": 2, "Dcut": 8, "steps": 20, "batch": 1, "field": False,
         "precision": "fp64", "fp64_steps": 2, "x6_steps": 0, "z2": False},
        # a 3D flow in the default precision up to its steady bond dimension 10
        {"name": "flow_3d_d10", "kind": "flow", "d": 3, "Dcut": 10, "steps": 7, "batch": 1, "field": False,
         "precision": "fp64", "fp64_steps": 2, "x6_steps": 0, "z2": False},
        # a temperature / field scan in one context with the mixed precision schedule
        {"name": "scan_4d_d5", "kind": "flow", "d": 4, "Dcut": 5, "steps": 9, "batch": 16, "field": True,
         "precision": "fp16x3", "fp64_steps": 3, "x6_steps": 6, "z2": False},
        # energy and magnetisation of a 4D flow: forward and backward through torch.autograd
        {"name": "grad_4d_d5", "kind": "grad", "d": 4, "Dcut": 5, "steps": 5, "batch": 2, "mode": "eig"},
        # single steps in FP64: a small 4D one, one with unequal bond dimensions (rows that are no multiple of any
        # tile), the zero-field block-sparse form, and the largest Gram matrices the library takes (2D, 256 x 256)
        {"name": "step_4d_d4_fp64", "kind": "step", "dims": "4,4,4,4", "Dcut": 4, "axis": 3, "precision": "fp64",
         "z2": False},
        {"name": "step_4d_ragged_fp64", "kind": "step", "dims": "5,6,4,5", "Dcut": 6, "axis": 1,
         "precision": "fp64", "z2": False},
        {"name": "step_4d_d6_fp64_z2", "kind": "step", "dims": "6,6,6,6", "Dcut": 6, "axis": 0, "precision": "fp64",
         "z2": True},
        {"name": "step_2d_d16_fp64", "kind": "step", "dims": "16,16", "Dcut": 16, "axis": 1, "precision": "fp64",
         "z2": False},
        # single steps in split precision: six products on unequal bond dimensions, three fp16 products at 8^4
        {"name": "step_4d_ragged_bf16x6", "kind": "step", "dims": "6,7,7,6", "Dcut": 7, "axis": 2,
         "precision": "bf16x6", "z2": False},
        {"name": "step_4d_d8_fp16x3", "kind": "step", "dims": "8,8,8,8", "Dcut": 8, "axis": 3,
         "precision": "fp16x3", "z2": False},
        # the paper's scale: the next steady step of a zero-field 4D flow at bond dimension 10
        {"name": "steady_4d_d10_fp16x3_z2", "kind": "steady", "Dcut": 10, "precision": "fp16x3",
         "beta": 0.1497},
        # the squeeze's product on its own, at the shape of one chunk of a 7^4 step
        {"name": "gemm_d7_fp16x3", "kind": "gemm", "M": 2401, "N": 16807, "K": 2401, "npass": 3, "fp16": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("flow", "flow", "grad", "step", "step", "step", "split", "split", "gemm", "gemm", "steady"))
    if kind == "flow":
        d = rng.choice((2, 3, 4))
        dcut = rng.choice(CLEAN_DCUT[d])
        batch = rng.choice((1, 1, 2, 5, 16)) if dcut < 10 else 1
        mixed = d == 4 and dcut == 5 and rng.random() < 0.6
        if d == 4 and not mixed:
            batch = min(batch, 5)
        top = {2: 24, 3: 7 if dcut == 10 else 15, 4: 9 if mixed or batch == 1 else 5}[d]
        field = rng.random() < 0.5
        return {"kind": "flow", "d": d, "Dcut": dcut, "steps": rng.randint(max(4, top - 4), top), "batch": batch,
                "field": field, "precision": rng.choice(("fp16x3", "bf16x3", "bf16x6")) if mixed else "fp64",
                "fp64_steps": 3, "x6_steps": rng.choice((0, 6)) if mixed else 0,
                "z2": not field and rng.random() < 0.5}
    if kind == "grad":
        d = rng.choice((2, 3, 4))
        dcut = {2: rng.choice((4, 6, 8)), 3: rng.choice((4, 5, 6)), 4: rng.choice((3, 5))}[d]
        return {"kind": "grad", "d": d, "Dcut": dcut, "steps": rng.randint(4, 5 if d == 4 else 9),
                "batch": rng.randint(1, 2), "mode": rng.choice(("eig", "fixed"))}
    if kind in ("step", "split"):
        # FP64 steps up to about 1e12 flops, split-precision ones up to the 8^4 step; split modes use the tensor
        # cores from 256 rows on
        while True:
            d = rng.choice((2, 3, 4, 4))
            z2 = rng.random() < 0.4
            dims = [rng.randint(3, {2: 16, 3: 12, 4: 8}[d]) for _ in range(d)]
            dcut = min(16, max(dims) + rng.randint(0, 2))
            c = {"kind": "step", "dims": ",".join(map(str, dims)), "Dcut": dcut, "axis": rng.randrange(d),
                 "precision": "fp64" if kind == "step" else rng.choice(("fp16x3", "fp16x3", "bf16x3", "bf16x4",
                                                                         "bf16x6")), "z2": z2}
            f = _step_flops(dims, c["axis"], dcut) * (0.25 if z2 else 1.0)
            if f <= (1e12 if kind == "step" else 7.1e13) and (kind == "step" or math.prod(dims) >= 256):
                return c
    if kind == "steady":
        return {"kind": "steady", "Dcut": 10, "precision": rng.choice(("fp16x3", "bf16x3", "fp16x4")),
                "beta": round(rng.uniform(0.149, 0.151), 5)}
    return {"kind": "gemm", "M": _log_int(rng, 128, 4100), "N": _log_int(rng, 256, 33000),
            "K": _log_int(rng, 64, 4100), "npass": rng.choice((1, 3, 4)), "fp16": True} if rng.random() < 0.5 else \
        {"kind": "gemm", "M": _log_int(rng, 128, 4100), "N": _log_int(rng, 256, 33000), "K": _log_int(rng, 64, 4100),
         "npass": rng.choice((1, 3, 4, 6)), "fp16": False}


# ------------------------------------------------------------------------------------------------- inputs
def _temperatures(case, seed):
    """The (beta, h) instances of a flow: temperatures around the transition, h = 0 or a small field."""
    rng = np.random.default_rng(seed)
    lo, hi = BETA[case["d"]]
    n = case["batch"]
    beta = np.sort(rng.uniform(lo, hi, n))
    if case["kind"] == "grad":
        return beta, rng.uniform(0.005, 0.02, n)
    if not case["field"]:
        return beta, np.zeros(n)
    return beta, rng.choice((0.0, 1e-5, 1e-3), n) if n > 1 else np.full(1, 1e-3)


def _dims(case):
    return tuple(int(x) for x in case["dims"].split(","))


def _evens(dims):
    return tuple((n + 1) // 2 for n in dims)


def _site_tensor(case, seed):
    """A site tensor as a flow holds it: entries that decay with every bond index from a dominant one, generic
    otherwise (no degenerate spectra); with the zero-field block structure for z2 (values of each bond even-parity
    first)."""
    dims = _dims(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    T = torch.randn(dims + dims, generator=g, device="cuda", dtype=torch.float64) * 0.3
    T[(0,) * (2 * len(dims))] = 1.0
    odd = torch.zeros((), dtype=torch.int64, device="cuda")
    for axis in range(2 * len(dims)):
        n = dims[axis % len(dims)]
        i = torch.arange(n, device="cuda")
        e = _evens(dims)[axis % len(dims)] if case["z2"] else n
        shape = [1] * (2 * len(dims))
        shape[axis] = n
        # even values 0, 2, 4, ... and odd values 1, 3, ... of the decay, stored even first
        level = torch.where(i < e, 2 * i if case["z2"] else i, 2 * (i - e) + 1)
        T *= torch.pow(0.5, level.double()).reshape(shape)
        odd = odd + (i >= e).long().reshape(shape)
    if case["z2"]:
        T = torch.where(odd % 2 == 0, T, torch.zeros_like(T))
    return (T / T.norm()).cpu().numpy()


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    if kind == "flow":
        beta, h = _temperatures(case, seed)
        return {"case": case, "beta": beta, "h": h, "stream": stream}
    if kind == "grad":
        beta, h = (torch.tensor(x, dtype=torch.float64, requires_grad=True) for x in _temperatures(case, seed))
        return {"case": case, "beta": beta, "h": h}
    if kind == "step":
        T = _site_tensor(case, seed)
        flow = HOTRG(len(_dims(case)), 0.3, 0.0, case["Dcut"], precision=case["precision"], fp64_steps=0,
                     z2=case["z2"], stream=stream)
        flow.set_tensor(T, evens=_evens(_dims(case)) if case["z2"] else None)
        return {"case": case, "flow": flow, "checkpoint": flow.state_save()}
    if kind == "steady":
        rng = np.random.default_rng(seed)
        beta = case["beta"] + float(rng.uniform(-2e-4, 2e-4))
        return {"case": case, "beta": beta, "stream": stream, **_start_flow(case, beta, stream)}
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    A = torch.randn((case["M"], case["K"]), generator=g, device="cuda")
    Bt = torch.randn((case["N"], case["K"]), generator=g, device="cuda")
    return {"case": case, "A": A, "Bt": Bt}


def _start_flow(case, beta, stream):
    """A zero-field 4D flow that has reached its steady bond dimensions (three steps)."""
    flow = HOTRG(4, beta, 0.0, case["Dcut"], precision=case["precision"], z2=True, stream=stream)
    for _ in range(3):
        flow.step()
    return {"flow": flow, "steps": 3}


# ------------------------------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "flow":
        out = []
        with HOTRG(case["d"], state["beta"], state["h"], case["Dcut"], precision=case["precision"],
                   fp64_steps=case["fp64_steps"], x6_steps=case["x6_steps"], z2=case["z2"],
                   stream=state["stream"]) as flow:
            for _ in range(case["steps"]):
                flow.step()
                out.append(flow.free_energy()[0])
            lnc = [flow.ln_norms(i) for i in range(flow.batch)]
            x = [flow.observables(i)["x_indicator"] for i in range(flow.batch)]
        kept = np.float64 if case["precision"] == "fp64" else np.float32
        return {"lnz": np.array(out, dtype=kept), "ln_norms": np.array(lnc, dtype=kept), "x": np.array(x, dtype=kept)}
    if kind == "grad":
        y = lnz_autograd(state["beta"], state["h"], d=case["d"], Dcut=case["Dcut"], nsteps=case["steps"],
                         mode=case["mode"])
        db, dh = torch.autograd.grad(y.sum(), (state["beta"], state["h"]))
        return {"lnz": y.detach(), "db": db, "dh": dh}
    if kind == "step":
        flow = state["flow"]
        flow.state_load(state["checkpoint"])
        flow.step(case["axis"])
        lnz = flow.free_energy()[0]
        T = flow.get_tensor()
        if case["precision"] != "fp64":
            lnz, T = lnz.astype(np.float32), T.astype(np.float32)
        return {"lnz": lnz, "tensor": T}
    if kind == "steady":
        if state["steps"] >= 60:  # a flow ends at 64 steps: start the next one
            state["flow"].close()
            state.update(_start_flow(case, state["beta"], state["stream"]))
        flow = state["flow"]
        flow.step()
        state["steps"] += 1
        ob = flow.observables()
        spectra = [flow.spectra(ob["steps"], b) for b in range(4) if b != ob["last_axis"]]
        return {"lnz": np.float32(ob["lnz_per_site"]), "ln_c": np.float32(ob["last_ln_c"]),
                "x": np.float32(ob["x_indicator"]), "spectra": np.array(spectra, dtype=np.float32)}
    return gemm_split(state["A"], state["Bt"], npass=case["npass"], fp16=case["fp16"])


# ------------------------------------------------------------------------------------------------- work
def _step_flops(dims, axis, dcut):
    """2 prod(chi) P^3: the squeeze of one step."""
    f = 2.0 * math.prod(dims) ** 3
    for b, n in enumerate(dims):
        if b != axis:
            f *= min(n * n, dcut)
    return f


def _flow_work(d, dcut, steps):
    dims, flops, nbytes = [2] * d, 0.0, 0.0
    for n in range(steps):
        a = d - 1 - n % d
        flops += _step_flops(dims, a, dcut)
        nbytes += 8.0 * math.prod(dims) ** 2
        dims = [x if b == a else min(x * x, dcut) for b, x in enumerate(dims)]
        nbytes += 8.0 * math.prod(dims) ** 2
    return nbytes, flops


def work(case):
    """The tensors read and written once by every step, and the flops of the squeezes (a quarter of the dense
    count with the zero-field block structure; five times it with both tangents)."""
    kind = case["kind"]
    if kind in ("flow", "grad"):
        nbytes, flops = _flow_work(case["d"], case["Dcut"], case["steps"])
        tangents = kind == "grad"
        flops *= case["batch"] * (5 if tangents else 1) * (0.25 if case.get("z2") else 1)
        return {"bytes": nbytes * case["batch"] * (3 if tangents else 1), "flops": flops}
    if kind == "step":
        dims = _dims(case)
        new = [n if b == case["axis"] else min(n * n, case["Dcut"]) for b, n in enumerate(dims)]
        return {"bytes": 8.0 * (math.prod(dims) ** 2 + math.prod(new) ** 2),
                "flops": _step_flops(dims, case["axis"], case["Dcut"]) * (0.25 if case["z2"] else 1)}
    if kind == "steady":
        return {"bytes": 16.0 * case["Dcut"] ** 8, "flops": 0.5 * case["Dcut"] ** 15}
    return {"bytes": 4.0 * (case["M"] * case["K"] + case["N"] * case["K"] + case["M"] * case["N"]),
            "flops": 2.0 * case["M"] * case["N"] * case["K"]}


# ------------------------------------------------------------------------------------------------- 64-bit values
def _isometry(G, n, dcut, evens):
    """Leading eigenvectors of G (n^2 x n^2), descending, largest component positive; with evens, those of even
    parity first."""
    lam, V = torch.linalg.eigh(G)
    lam, V = lam.flip(0), V.flip(1)
    chi = min(n * n, dcut)
    V = V[:, :chi].clone()
    top = V.abs().argmax(0)
    V = V * torch.sign(V[top, torch.arange(chi, device=V.device)])
    if evens is not None:
        par = (torch.arange(n, device=V.device) >= evens).long()
        odd = ((par[:, None] + par[None, :]) % 2).reshape(-1)[top]
        V = torch.cat((V[:, odd == 0], V[:, odd == 1]), 1)
    return V.T.reshape(chi, n, n)


def _step64(T, axis, dcut, evens=None):
    """One coarse-graining step (before normalisation) in FP64."""
    d = T.dim() // 2
    trans = [b for b in range(d) if b != axis]
    U = {}
    for b in trans:
        n, m = T.shape[b], T.shape[axis]
        Q = []
        for other in (d + axis, axis):
            X = T.movedim((b, other), (0, 1)).reshape(n * m, -1)
            Q.append((X @ X.T).reshape(n, m, n, m))
        G = torch.einsum("iajb,kalb->ikjl", Q[0], Q[1]).reshape(n * n, n * n)
        U[b] = _isometry(G, n, dcut, None if evens is None else evens[b])
    nd = [U[b].shape[0] if b in U else T.shape[b] for b in range(d)]
    new = torch.empty(nd + nd, dtype=T.dtype, device=T.device)
    P = math.prod(T.shape[:d])
    B = T.movedim(axis, d - 1).reshape(P, P)  # rows: the transverse unprimed legs, then u_axis; columns: primed
    for ks in itertools.product(*[range(U[b].shape[0]) for b in trans]):
        X = T
        for b, k in zip(trans, ks):
            X = torch.tensordot(U[b][k], X, dims=([0], [b])).movedim(0, b)
        # site 1: contract (transverse legs, p_axis) with site 2's (transverse legs, u_axis)
        order = [axis] + [d + b for b in range(d) if b != axis] + trans + [d + axis]
        O = X.permute(order).reshape(-1, P) @ B
        O = O.reshape([T.shape[axis]] + [T.shape[b] for b in trans] + list(T.shape[:d]))
        # axes: u_axis of site 1, the transverse primed legs of site 1, the primed legs of site 2
        at, names = len(trans), list(range(d))
        for b in trans:
            pos = 1 + names.index(b) + at  # this leg of site 2
            O = torch.tensordot(O, U[b], dims=([1, pos], [1, 2]))
            O = O.movedim(-1, pos - 1)
            at -= 1
        idx = [None] * d
        for b, k in zip(trans, ks):
            idx[b] = k
        new[tuple(slice(None) if i is None else i for i in idx)] = O
    return new


def _initial64(d, beta, h):
    W = torch.tensor([[math.sqrt(math.cosh(beta)), s * math.sqrt(math.sinh(beta))] for s in (1.0, -1.0)],
                     dtype=torch.float64)
    T = 0.0
    for s, w in zip((1.0, -1.0), W):
        t = torch.tensor(math.exp(beta * h * s), dtype=torch.float64)
        for _ in range(2 * d):
            t = t[..., None] * w
        T = T + t
    return T.cuda()


def _flow64(d, beta, h, dcut, steps):
    """(ln Z/N after every step, ln c_0.., X of the last step)"""
    T = _initial64(d, beta, h)
    lnc, total, lnz = [], 0.0, []
    for n in range(steps + 1):
        if n:
            axis = d - 1 - (n - 1) % d
            T = _step64(T, axis, dcut)
        c = float(T.norm())
        T = T / c
        lnc.append(math.log(c))
        total += math.log(c) / 2 ** n
        P = math.prod(T.shape[:d])
        lnz.append(total + math.log(float(torch.trace(T.reshape(P, P)))) / 2 ** n)
    n = T.shape[axis]
    M = T.movedim((axis, d + axis), (0, 1)).reshape(n, n, P // n, P // n).diagonal(dim1=2, dim2=3).sum(-1)
    return lnz[1:], lnc, float(torch.trace(M) ** 2 / torch.trace(M @ M))


def exact(case, seed):
    kind = case["kind"]
    if kind == "flow":
        beta, h = _temperatures(case, seed)
        got = [_flow64(case["d"], b, x, case["Dcut"], case["steps"]) for b, x in zip(beta, h)]
        return {"lnz": np.array([g[0] for g in got]).T.copy(), "ln_norms": np.array([g[1] for g in got]),
                "x": np.array([g[2] for g in got])}
    if kind == "grad":
        # ln Z/N; its derivatives have no closed 64-bit form here (difference quotients are less exact)
        beta, h = _temperatures(case, seed)
        return {"lnz": np.array([_flow64(case["d"], b, x, case["Dcut"], case["steps"])[0][-1]
                                 for b, x in zip(beta, h)]), "db": None, "dh": None}
    if kind == "step":
        dims = _dims(case)
        if _step_flops(dims, case["axis"], case["Dcut"]) > 1.2e13:
            return None
        T = torch.from_numpy(_site_tensor(case, seed)).cuda()
        new = _step64(T, case["axis"], case["Dcut"], _evens(dims) if case["z2"] else None)
        c = float(new.norm())
        new = (new / c).cpu().numpy()
        P = math.prod(new.shape[:len(dims)])
        # the accumulator still holds ln c_0 of the context's own initial tensor
        lnc0 = math.log(float(_initial64(len(dims), 0.3, 0.0).norm()))
        return {"lnz": np.array([lnc0 + 0.5 * math.log(c) + 0.5 * math.log(np.trace(new.reshape(P, P)))]),
                "tensor": new}
    if kind == "steady":
        return None
    s = prepare(case, seed)
    return s["A"].double() @ s["Bt"].double().T
