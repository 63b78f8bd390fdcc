"""Timed cases of the library: what a user's program has it do, through the binding's entry points.

A program of this library assembles the coupling matrix of a coil column by column, compresses the
columns in Tucker form (truncated HOSVD or the randomized range finder), tunes the handle for its
number of right-hand sides and then calls the two products many times.  The cases are these calls:
the forward and the adjoint product from the smallest grid to the 1 mm one, both products of
ACA storage and of a coil close to the voxels, and the two compressors.

`kind` is what run() does: "forward" (Y = Z X), "adjoint" (Psi = Z^H Phi), "step" (both, as one
solver iteration does) or "compress" (the columns to a handle, whose ranks and columns come back).
`coil` names the workload of inputs.py whose sources, frequency and mask the case takes.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2103_06393_gb300 import inputs, zbc

PREC = {"fp32": zbc.FP32_SIMT, "auto": zbc.AUTO}
RADIUS = {"tiny": 0.15, "precision": 0.14, "batching": 0.16, "learned": 0.12, "large": 0.30}


def listed():
    return [
        # the smallest call: one vector through the smoke-sized handle, with the default arithmetic;
        # latency and launches are all of it
        _case("tiny_forward", "forward", "tiny", (24, 24, 24), 64, 1, tol=1e-8, method="hosvd", prec="fp32", rank=13),
        # the same handle's adjoint after tuning
        _case("tiny_adjoint", "adjoint", "tiny", (24, 24, 24), 64, 1, tol=1e-8, method="hosvd", rank=13),
        # a head coil at 2 mm with 16 right-hand sides, as a solver's block of port excitations
        _case("head_forward", "forward", "precision", (96, 96, 96), 1024, 16, tol=1e-6, rank=11),
        _case("head_adjoint", "adjoint", "precision", (96, 96, 96), 1024, 16, tol=1e-6, rank=11),
        # a 16-loop coil around a masked 1.5 mm grid: many right-hand sides at once, then few
        _case("body_forward", "forward", "batching", (160, 160, 128), 512, 32, tol=1e-6, rank=10),
        _case("body_adjoint", "adjoint", "batching", (160, 160, 128), 512, 4, tol=1e-6, rank=10),
        # the 1 mm grid (a part of its coil's segments): the largest vectors
        _case("fine_forward", "forward", "large", (320, 320, 256), 128, 8, tol=1e-5, rank=7),
        _case("fine_adjoint", "adjoint", "large", (320, 320, 256), 128, 8, tol=1e-5, rank=7),
        # sources two voxels from the grid (a surface coil), odd sizes: one solver iteration
        _case("near_step", "step", "learned", (101, 117, 96), 128, 8, tol=1e-6, rank=15),
        # Z = U V^H by ACA with U in Tucker form (Algorithm 3's storage): one solver iteration
        _case("aca_step", "step", "large", (64, 48, 40), 512, 3, tol=1e-3, storage="aca", rank=9),
        # the truncated HOSVD of assembled columns, the paper's compressor
        _case("hosvd", "compress", "precision", (96, 96, 96), 8, 8, tol=1e-6, method="hosvd", rank=11),
        # the randomized compressor at the larger size it is used for
        _case("randomized", "compress", "learned", (128, 128, 128), 16, 16, tol=1e-6, rank=17),
    ]


def _case(name, kind, coil, n, M, p, tol, method="randomized", prec="auto", storage="tucker", q=3, rank=10, h=0.0):
    c = dict(kind=kind, coil=coil, n1=n[0], n2=n[1], n3=n[2], h=h, M=M, p=p, q=q, tol=tol, method=method, prec=prec,
             storage=storage, rank=rank)
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "adjoint", "adjoint", "step", "compress"])
    coil = rng.choice(["precision", "batching", "large", "learned"])
    if kind == "compress":
        method = rng.choice(["hosvd", "randomized"])
        n = [2 * _log_int(rng, 12, 48 if method == "hosvd" else 64) for _ in range(3)]
        M = rng.randint(2, 8)
        p, prec, storage, q = M, "auto", "tucker", 3
    else:
        method = "randomized"
        n = [_log_int(rng, 24, 320) for _ in range(3)]
        while n[0] * n[1] * n[2] > 12e6:
            n[rng.randrange(3)] = _log_int(rng, 24, 160)
        nv = n[0] * n[1] * n[2]
        storage = "aca" if nv < 2e5 and rng.random() < 0.5 else "tucker"
        q = 12 if nv < 1e6 and storage == "tucker" and rng.random() < 0.25 else 3
        M = _log_int(rng, 64, 1024)
        p = _log_int(rng, 1, 64)
        prec = rng.choice(["auto", "auto", "auto", "fp32"])
        M = max(16, min(M, int(1.0e9 * 3 / (nv * q))))
        p = max(1, min(p, int(2.0e10 * 3 / (nv * M * q)) - 8, int(6e8 / (nv * q))))
    # the voxel size that makes the grid's wider transverse side reach 0.62 of the coil's radius
    # (0.55 inside the nearest of the random sources)
    h = 2.0 * (0.55 if coil == "learned" else 0.62) * RADIUS[coil] / max(n[0], n[1])
    return _case(None, kind, coil, n, M, p, tol=rng.choice([1e-5, 1e-6]) if storage == "tucker" else 1e-3,
                 method=method, prec=prec, storage=storage, q=q, rank=10, h=h)


# ---------------------------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------------------------

def _geometry(c, seed, count, even):
    """The grid (its sizes rounded up to even ones if asked for: the compressors take those) and
    `count` of the coil's segments, drawn from the seed."""
    w = inputs.workload(c["coil"])
    n = [c["n1"], c["n2"], c["n3"]]
    n = [x + x % 2 for x in n] if even else n
    g = dataclasses.replace(w.grid, n1=n[0], n2=n[1], n3=n[2], h=c["h"] or w.grid.h)
    if c["h"]:
        g = dataclasses.replace(g, mask_box=0.0)
    rng = np.random.default_rng([seed, 1])
    if c["coil"] == "learned":
        segs = inputs.random_cylinder_segments(g, count, seed=seed, z_half=0.6 * g.n3 * g.h)
    else:
        segs = w.segments.subset(np.sort(rng.choice(w.segments.m, size=min(count, w.segments.m), replace=False)))
    return w, g, segs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _cn01(gen, cols, rows):
    return torch.randn((cols, rows), dtype=torch.complex64, device="cuda", generator=gen)


def _assemble(c, g, segs, freq, dtype):
    ds = zbc.DeviceSegments(segs)
    Z = zbc.colmajor(c["q"] * g.nv, segs.m, dtype)
    idx = torch.arange(segs.m, dtype=torch.int32, device="cuda")
    return zbc.vsie_assemble_columns_op(g, ds, freq, idx, Z, q=c["q"])


def _sketches(c, g, seed):
    gen = _gen(seed + 7)
    n1, n2, n3 = g.shape
    return [_cn01(gen, 32, r) for r in (n2 * n3, n1 * n3, n1 * n2)]


def _compress(c, g, Z, sk):
    if c["method"] == "hosvd":
        return zbc.tucker_compress(Z, g, c["tol"], q=c["q"])[0]
    model = zbc.rank_model(sk, 32, fixed_width=32)
    return zbc.tucker_compress(Z, g, c["tol"], q=c["q"], method=zbc.RANDOMIZED_FIXED, model=model)[0]


def _mirrored(tensors, g, M):
    """The first M columns of the mirror images (in x, y and z) of the compressed ones: the field
    of a source mirrored in axis d is the mirrored field with its component d reversed.  The coils
    are symmetric, so the images are their segments too, and an eighth of the columns is compressed.
    For the piecewise-linear basis (12 row blocks 3 l + k) the slope along d changes its sign too."""
    out = []
    for image in range(8):
        flip = [d for d in range(3) if image >> d & 1]
        for col in tensors:
            if len(out) == M:
                return out
            new = []
            for b, (G, U) in enumerate(col):
                sign = 1
                for d in flip:
                    sign *= (-1 if b % 3 == d else 1) * (-1 if b // 3 == d + 1 else 1)
                new.append((sign * G, [u[::-1] if d in flip else u for d, u in enumerate(U)]))
            out.append(new)
    return out


def _cut(tensors, n):
    """The tensors on the first n1 x n2 x n3 voxels, factors orthonormal again."""
    def one(G, U):
        new = []
        for d, u in enumerate(U):
            if u.shape[0] > n[d]:
                u, r = np.linalg.qr(u[:n[d]])
                G = np.moveaxis(np.tensordot(r, G, axes=(1, d)), 0, d)
            new.append(u)
        return G, new

    return [[one(*t) for t in col] for col in tensors]


def _handle(c, seed):
    """The compressed matrix on the case's grid."""
    if c["storage"] == "aca":
        w, g, segs = _geometry(c, seed, c["M"], even=True)
        h = zbc.aca_compress(g, zbc.DeviceSegments(segs), w.freq_hz, c["tol"], 96, mode=zbc.ACA_DENSE_U)[0]
        tensors, V = h.tensors()
    else:
        w, g, segs = _geometry(c, seed, -(-c["M"] // 8), even=True)
        small = None
        per = max(1, int(4e9 / (8 * c["q"] * g.nv)))
        sk = _sketches(c, g, seed)
        for at in range(0, segs.m, per):  # columns in batches, as the memory allows
            part = segs.subset(np.arange(at, min(segs.m, at + per)))
            Z = _assemble(c, g, part, w.freq_hz, torch.complex64)
            if small is None:
                small = _compress(c, g, Z, sk)
            else:
                small = zbc.tucker_compress(Z, g, c["tol"], q=c["q"], method=zbc.RANDOMIZED_FIXED,
                                            model=zbc.rank_model(sk, 32, fixed_width=32), append_to=small)[0]
            del Z
        tensors, V = _mirrored(small.tensors()[0], g, c["M"]), None
    n = (c["n1"], c["n2"], c["n3"])
    if g.shape != n:
        tensors = _cut(tensors, n)
        g = dataclasses.replace(g, n1=n[0], n2=n[1], n3=n[2])
    return g, zbc.zbc_create_from_host(g, c["q"], tensors, V)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "compress":
        w, g, segs = _geometry(c, seed, c["M"], even=True)
        Z = _assemble(c, g, segs, w.freq_hz, torch.complex128)
        return dict(c=c, g=g, Z=Z, sk=_sketches(c, g, seed), X=torch.eye(c["M"], dtype=torch.complex64, device="cuda"),
                    Y=zbc.colmajor(c["q"] * g.nv, c["M"], torch.complex64))
    g, h = _handle(c, seed)
    m, rows, gen = h.info().m, c["q"] * g.nv, _gen(seed)
    s = dict(c=c, g=g, h=h, prec=PREC[c["prec"]])
    if c["prec"] == "auto":
        zbc.zbc_tune(h, c["p"])
    if c["kind"] != "adjoint":
        s.update(X=_cn01(gen, c["p"], m), Y=zbc.colmajor(rows, c["p"], torch.complex64))
    if c["kind"] != "forward":
        s.update(Phi=_cn01(gen, c["p"], rows), Psi=zbc.colmajor(m, c["p"], torch.complex64))
    return s


def run(s):
    if s["c"]["kind"] == "compress":
        h = _compress(s["c"], s["g"], s["Z"], s["sk"])
        return {"ranks": h.export()[0], "columns": zbc.zbc_matvec(h, s["X"], s["Y"])}
    out = {}
    if "X" in s:
        out["Y"] = zbc.zbc_matvec(s["h"], s["X"], s["Y"], s["prec"])
    if "Phi" in s:
        out["Psi"] = zbc.zbc_rmatvec(s["h"], s["Phi"], s["Psi"], s["prec"])
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without, and its results in 64 bits
# ---------------------------------------------------------------------------------------------

def work(case):
    c = case
    nv, r, q, M, p = c["n1"] * c["n2"] * c["n3"], c["rank"], c["q"], c["M"], c["p"]
    stored = q * M * (r ** 3 + (c["n1"] + c["n2"] + c["n3"]) * r)
    if c["kind"] == "compress":  # the columns once, the tensors and the returned columns once
        return {"bytes": 16.0 * q * nv * M + 8.0 * stored + 8.0 * q * nv * M, "flops": 8.0 * q * nv * M * r}
    if c["storage"] == "aca":
        stored = q * 96 * (r ** 3 + (c["n1"] + c["n2"] + c["n3"]) * r) + 96 * M
    products = 2 if c["kind"] == "step" else 1  # each stored value meets each right-hand side
    return {"bytes": products * 8.0 * (stored + M * p + q * nv * p), "flops": products * 8.0 * p * stored}


def _dense(col, b, dev="cuda"):
    """Row block b of a column from its Tucker tensor, (n3, n2, n1) flattened, in 64 bits."""
    G, (U1, U2, U3) = col[b]
    G, U1, U2, U3 = (torch.from_numpy(np.ascontiguousarray(x)).to(dev, torch.complex128) for x in (G, U1, U2, U3))
    T = torch.einsum("abc,kc->kab", G, U3)
    T = torch.einsum("kab,jb->kja", T, U2)
    return (T.reshape(-1, T.shape[2]) @ U1.T).reshape(-1)


def exact(case, seed):
    s = prepare(case, seed)
    c, g = s["c"], s["g"]
    if c["kind"] == "compress":
        Z = s["Z"]
        if c["method"] == "hosvd":
            Z = torch.stack([torch.cat([_truncated(b, g, c["tol"]) for b in col.reshape(c["q"], g.nv)]) for col in Z])
        return {"ranks": None, "columns": Z}  # what the randomized compressor approximates to tol
    tensors, V = s["h"].tensors()
    V = None if V is None else torch.from_numpy(np.ascontiguousarray(V)).cuda().to(torch.complex128)
    del s["h"]
    M, out, step = len(tensors), {}, 16
    if "X" in s:
        X = s["X"].to(torch.complex128)
        X = X if V is None else X @ V.conj()  # X' = V^H X, a row per right-hand side
        Y = torch.zeros_like(s["Y"], dtype=torch.complex128)
    if "Phi" in s:
        Phi = s["Phi"].to(torch.complex128)
        Psi = torch.zeros((c["p"], M), dtype=torch.complex128, device="cuda")
    for b in range(c["q"]):
        rows = slice(b * g.nv, (b + 1) * g.nv)
        for j in range(0, M, step):
            Z = torch.stack([_dense(col, b) for col in tensors[j:j + step]])
            if "X" in s:
                Y[:, rows].addmm_(X[:, j:j + step], Z)
            if "Phi" in s:
                Psi[:, j:j + step].addmm_(Phi[:, rows], Z.conj().T)
    if "X" in s:
        out["Y"] = Y
    if "Phi" in s:
        out["Psi"] = Psi if V is None else Psi @ V.T
    return out


def _truncated(a, g, tol):
    """The truncated HOSVD of one tensor: per mode the smallest rank whose tail is within tol^2 / 3."""
    A = a.reshape(g.n3, g.n2, g.n1)
    total, B = float(torch.linalg.vector_norm(A)) ** 2, A
    for d in range(3):
        F = torch.movedim(A, d, 0).reshape(A.shape[d], -1)
        w, v = torch.linalg.eigh(F @ F.conj().T)
        tail = torch.cumsum(w.clamp(min=0), 0)  # ascending: the sums of the smallest
        U = v[:, int((tail <= tol * tol / 3 * total).sum()):]
        B = torch.movedim(torch.tensordot(U @ U.conj().T, B, dims=([1], [d])), 0, d)
    return B.reshape(-1)
