"""The workloads the library is timed on: what its users call, over the sizes, types and options they call it with.

A case is one call of a public entry point on operands that are already on the GPU:

* ``kron2`` / ``kron3``: ``Y <- alpha (A (x) B [(x) C]) X + beta Y`` with components of ``m`` x ``n`` (``n`` nodes in,
  ``m`` nodes out on every axis), ``batch`` instances, ``dtype`` storage and ``compute`` arithmetic; ``trans`` is the
  op of every component, ``transx`` the op of X (2-D), ``pad`` the elements by which the leading dimensions exceed
  the smallest ones;
* ``varlen``: one ``VarlenPlan.execute`` over ``batch`` instances, 2-D and 3-D mixed (a share ``p3`` in 3-D),
  every n in ``nmin..nmax`` equally often, in random order, one component set per (kind, n).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1304_7054_gb300 as kg

DTYPES = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16, "f16": torch.float16,
          "c64": torch.complex64, "c128": torch.complex128}
BYTES = {"f32": 4, "f64": 8, "bf16": 2, "f16": 2, "c64": 8, "c128": 16}


def _kron(kind, n, batch, dtype="f32", compute="native", m=None, alpha=1.0, beta=0.0, trans="N", transx="N", pad=0,
          name=None):
    c = {"entry": f"kron{kind}", "kind": kind, "m": m or n, "n": n, "batch": batch, "dtype": dtype,
         "compute": compute, "alpha": alpha, "beta": beta, "trans": trans, "transx": transx, "pad": pad}
    return dict(c, name=name) if name else c


def _varlen(batch, dtype="f32", nmin=4, nmax=16, p3=0.5, name=None):
    c = {"entry": "varlen", "batch": batch, "dtype": dtype, "nmin": nmin, "nmax": nmax, "p3": p3}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: 1024 low-order 2-D elements, where latency is all there is
        _kron(2, 4, 1 << 10, name="kron2-f32-n4-b1024"),
        # the headline workload: 2^20 2-D operands at n = 16
        _kron(2, 16, 1 << 20, name="kron2-f32-n16"),
        # an operator added to a right-hand side (y += A x), odd order, a batch that no tile divides
        _kron(2, 9, 999_983, alpha=-1.0, beta=1.0, name="kron2-f32-n9-accumulate"),
        # the 3-D action at n = 16
        _kron(3, 16, 1 << 16, name="kron3-f32-n16"),
        # the 3-D action in double precision
        _kron(3, 10, 1 << 16, dtype="f64", name="kron3-f64-n10"),
        # interpolation from 8 nodes to 12 quadrature points on every axis: rectangular components
        _kron(3, 8, 100_003, m=12, name="kron3-f32-8to12"),
        # row-major operands in a padded array (op(X) = X^T), as a C or PyTorch program stores its matrices
        _kron(2, 16, 1 << 18, transx="T", pad=4, name="kron2-f32-n16-rowmajor"),
        # 16-bit storage with FP32 arithmetic
        _kron(2, 8, 1 << 20, dtype="bf16", name="kron2-bf16-n8"),
        # 16-bit storage through the split tensor-core path, 2-D and 3-D
        _kron(2, 12, 1 << 20, dtype="f16", compute="bf16x3", name="kron2-f16-n12-bf16x3"),
        _kron(3, 16, 1 << 16, dtype="bf16", compute="bf16x3", name="kron3-bf16-n16-bf16x3"),
        # complex data with Hermitian-transposed components (the adjoint of a complex operator)
        _kron(2, 16, 1 << 19, dtype="c64", trans="C", name="kron2-c64-n16-adjoint"),
        # a mesh of mixed order and dimension in one call
        _varlen(200_000, name="varlen-f32-200k"),
    ]


def _batch(rng, per, lo, hi):
    """Instances of `per` elements: the total spread over its logarithm between lo and hi elements."""
    total = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(1, min(int(total / per), hi // per))


def draw(rng):
    what = rng.choice(["small", "2d", "2d", "accumulate", "3d", "3d", "double", "rect", "rowmajor", "store16", "split",
                       "split16", "complex", "varlen"])
    n = rng.randint(3, 16)
    kind = rng.choice([2, 3])
    if what == "small":
        kind, n = rng.choice([2, 3]), rng.randint(2, 8)
        return _kron(kind, n, rng.randint(1, 4096))
    if what in ("2d", "3d"):
        kind = int(what[0])
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 28))
    if what == "accumulate":
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 27), alpha=rng.choice([1.0, -1.0, 0.5]), beta=1.0,
                     trans=rng.choice(["N", "T"]))
    if what == "double":
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 25), dtype="f64")
    if what == "rect":   # interpolation up (N) or its transpose, integration back down (T)
        m = min(16, n + rng.randint(1, 4))
        n = m - rng.randint(1, min(4, m - 2))
        batch = _batch(rng, m ** kind, 1 << 16, 1 << 27)
        if rng.random() < 0.5:
            return _kron(kind, n, batch, m=m)
        return _kron(kind, m, batch, m=n, trans="T")
    if what == "rowmajor":
        return _kron(2, n, _batch(rng, n * n, 1 << 16, 1 << 26), transx="T", pad=rng.choice([0, 0, 1, 4, 16 - n]))
    if what == "store16":
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 27), dtype=rng.choice(["bf16", "f16"]))
    if what in ("split", "split16"):
        dtype = "f32" if what == "split" else rng.choice(["bf16", "f16"])
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 28), dtype=dtype, compute="bf16x3")
    if what == "complex":
        trans = rng.choice(["N", "T", "C"])
        return _kron(kind, n, _batch(rng, n ** kind, 1 << 16, 1 << 26), dtype="c64", trans=trans)
    nmin = rng.randint(2, 8)
    return _varlen(int(math.exp(rng.uniform(math.log(1000), math.log(200_000)))), dtype=rng.choice(["f32", "bf16", "f16"]),
                   nmin=nmin, nmax=rng.randint(nmin, 16), p3=rng.choice([0.0, 0.5, 0.5, 1.0]))


def _shapes(c):
    """Leading dimensions and instance strides (elements) of X and Y, and their extents in storage order."""
    k, m, n, pad = c["kind"], c["m"], c["n"], c["pad"]
    ldx, ldy = n + pad, m + pad
    return ldx, ldx * n ** (k - 1), ldy, ldy * m ** (k - 1)


def _view(t, c, which):
    """The logical operands or results in a flat array: [batch, (mode 3,) mode 2, mode 1] of the stored arrays."""
    ldx, ldxp, ldy, ldyp = _shapes(c)
    e, ld, ldp = (c["n"], ldx, ldxp) if which == "X" else (c["m"], ldy, ldyp)
    if c["kind"] == 2:
        return t.as_strided((c["batch"], e, e), (ldp, ld, 1))
    return t.as_strided((c["batch"], e, e, e), (ldp, ld * e, ld, 1))


def _components(c, rng, kind, m, n):
    """Host components, uniform in [-1, 1], stored for op `trans`."""
    shape = (m, n) if c.get("trans", "N") == "N" else (n, m)
    out = []
    for _ in range(kind):
        M = rng.uniform(-1.0, 1.0, shape)
        if c["dtype"].startswith("c"):
            M = M + 1j * rng.uniform(-1.0, 1.0, shape)
            M = M.astype(np.complex64 if c["dtype"] == "c64" else np.complex128)
        else:
            M = M.astype(np.float64 if c["dtype"] == "f64" else np.float32)
        out.append(M)
    return out


def _normal(count, dtype, gen):
    t = DTYPES[dtype]
    if t in (torch.bfloat16, torch.float16):
        return torch.randn(count, device="cuda", generator=gen).to(t)
    return torch.randn(count, device="cuda", generator=gen, dtype=t)


def prepare(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if c["entry"] != "varlen":
        _, ldxp, _, ldyp = _shapes(c)
        comps = _components(c, rng, c["kind"], c["m"], c["n"])
        X = _normal(c["batch"] * ldxp, c["dtype"], gen)
        Y = _normal(c["batch"] * ldyp, c["dtype"], gen) if c["beta"] else torch.zeros(
            c["batch"] * ldyp, device="cuda", dtype=DTYPES[c["dtype"]])
        return {"case": c, "comps": comps, "X": X, "Y": Y}
    classes = [(k, n) for k in (2, 3) for n in range(c["nmin"], c["nmax"] + 1)]
    comps = [_components(c, rng, k, n, n) for k, n in classes]
    # every n equally often, a share p3 of each in 3-D, in random order
    i = rng.permutation(c["batch"])
    ns, j = c["nmin"] + i % (c["nmax"] - c["nmin"] + 1), i // (c["nmax"] - c["nmin"] + 1)
    kinds = 2 + (np.floor((j + 1) * c["p3"]) > np.floor(j * c["p3"]))
    class_of = ((kinds - 2) * (c["nmax"] - c["nmin"] + 1) + ns - c["nmin"]).astype(np.int32)
    sizes = ns.astype(np.int64) ** kinds
    off = np.concatenate([np.zeros(1, np.int64), np.cumsum(sizes)])
    X = _normal(int(off[-1]), c["dtype"], gen)
    Y = torch.zeros_like(X)
    plan = kg.VarlenPlan([(k, n, *ms) for (k, n), ms in zip(classes, comps)], class_of, off[:-1], off[:-1],
                         io=c["dtype"])
    return {"case": c, "classes": classes, "comps": comps, "class_of": class_of, "off": off[:-1], "X": X, "Y": Y,
            "plan": plan, "workspace": plan.alloc_workspace()}


def run(state):
    c, X, Y = state["case"], state["X"], state["Y"]
    if c["entry"] == "varlen":
        return state["plan"].execute(X, Y, state["workspace"])
    m, n, t = c["m"], c["n"], c["trans"]
    ldx, ldxp, ldy, ldyp = _shapes(c)
    if c["kind"] == 2:
        A, B = state["comps"]
        return kg.kron2_batched(A, B, X, Y, ma=m, na=n, mb=m, nb=n, batch=c["batch"], alpha=c["alpha"], beta=c["beta"],
                                transa=t, transb=t, transx=c["transx"], ldx=ldx, ldxp=ldxp, ldy=ldy, ldyp=ldyp,
                                compute=c["compute"])
    A, B, C = state["comps"]
    return kg.kron3_batched(A, B, C, X, Y, ma=m, na=n, mb=m, nb=n, mc=m, nc=n, batch=c["batch"], alpha=c["alpha"],
                            beta=c["beta"], transa=t, transb=t, transc=t, ldx=ldx, ldx2=ldx * n, ldxp=ldxp, ldy=ldy,
                            ldy2=ldy * m, ldyp=ldyp, compute=c["compute"])


def _flops(kind, m, n):
    """Multiply-adds of the mode-by-mode action, two operations each."""
    return 2.0 * sum(m ** (k + 1) * n ** (kind - k) for k in range(kind))


def work(case):
    c = case
    if c["entry"] == "varlen":
        ns = range(c["nmin"], c["nmax"] + 1)
        mean = lambda f: sum(f(n) for n in ns) / len(ns)  # noqa: E731
        p3 = c["p3"]
        elems = (1 - p3) * mean(lambda n: n ** 2) + p3 * mean(lambda n: n ** 3)
        flops = (1 - p3) * mean(lambda n: _flops(2, n, n)) + p3 * mean(lambda n: _flops(3, n, n))
        return {"bytes": 2.0 * BYTES[c["dtype"]] * elems * c["batch"], "flops": flops * c["batch"]}
    k, m, n = c["kind"], c["m"], c["n"]
    elems = n ** k + m ** k * (2 if c["beta"] else 1)
    scale = 4.0 if c["dtype"].startswith("c") else 1.0
    return {"bytes": float(BYTES[c["dtype"]]) * elems * c["batch"], "flops": scale * _flops(k, m, n) * c["batch"]}


def _wide(t):
    return t.to(torch.complex128 if t.is_complex() else torch.float64)


def _act(ms, x):
    """Every component on its mode: ms[0] on the last stored axis (mode 1), and so on."""
    for axis, M in enumerate(ms):
        x = torch.tensordot(x, M, dims=([x.dim() - 1 - axis], [1])).movedim(-1, x.dim() - 1 - axis)
    return x


def exact(case, seed):
    c = case
    s = prepare(c, seed)
    X, Y = s["X"], s["Y"]
    out = _wide(Y)
    if c["entry"] == "varlen":
        class_of = torch.from_numpy(s["class_of"]).cuda()
        off = torch.from_numpy(s["off"]).cuda()
        for i, ((k, n), ms) in enumerate(zip(s["classes"], s["comps"])):
            at = off[class_of == i]
            if not len(at):
                continue
            at = at[:, None] + torch.arange(n ** k, device="cuda")
            x = _wide(X[at]).view(-1, *([n] * k))
            ms = [torch.from_numpy(M).cuda().double() for M in ms]   # 2-D: A, B; 3-D: A, B, C
            out[at] = _act(ms[::-1], x).reshape(at.shape)
        return out
    ms = []
    for M in s["comps"]:
        M = _wide(torch.from_numpy(M).cuda())
        ms.append(M if c["trans"] == "N" else M.T if c["trans"] == "T" else M.conj().T.resolve_conj())
    xv, yv = _view(X, c, "X"), _view(out, c, "Y")
    step = max(1, (1 << 26) // max(c["m"], c["n"]) ** c["kind"])
    for p in range(0, c["batch"], step):
        x = _wide(xv[p:p + step])
        if c["transx"] == "T":
            x = x.transpose(1, 2)
        y = c["alpha"] * _act(ms[::-1], x)
        yv[p:p + step] = y + c["beta"] * yv[p:p + step] if c["beta"] else y
    return out
