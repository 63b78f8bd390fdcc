"""ZBC_AUTO at the edges of the joint form: handles that cannot take it (ranks above its bases' 64
vectors) keep the forms they had, its workspaces (and the FP32 forward's) keep their place, a device
without room for it still runs the products, and vectors and columns of any size FP32 holds (the column
sums run in FP32 up to 4 / 2 right-hand sides, forward / adjoint, and on the tensor cores from there on),
to FP32's accuracy; and its bounded waits, which end a product that cannot go on with a status."""
import numpy as np
import pytest

from oracle import products
from paper_2103_06393_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()
from paper_2103_06393_gb300 import zbc  # noqa: E402

RTOL = 1e-5  # what every form meets


def _orth(rng, n, r):
    return np.linalg.qr(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)))[0]


def _c64(a):
    return a.astype(np.complex64).astype(np.complex128)


def _shared(n, m, R, r, seed=0, q=3, norm=1.0):
    """m columns of q tensors of ranks r whose factors lie in common bases of R vectors a mode."""
    rng = np.random.default_rng(seed)
    tens = [[None] * q for _ in range(m)]
    for k in range(q):
        B = [_orth(rng, n[d], R[d]) for d in range(3)]
        for j in range(m):
            G = rng.standard_normal(r) + 1j * rng.standard_normal(r)
            G *= norm / np.linalg.norm(G)
            tens[j][k] = _c64(G), [_c64(B[d] @ _orth(rng, R[d], r[d])) for d in range(3)]
    return inputs.Grid(*n, 0.001), tens


def _rel(a, b):
    a = a.astype(np.complex128)
    return float(np.max(np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)))


def _run(h, g, A, fwd, prec=None, q=3):
    B = zbc.colmajor(q * g.nv if fwd else h.info().m, A.shape[1], torch.complex64)
    B.fill_(float("nan"))
    call = zbc.zbc_matvec if fwd else zbc.zbc_rmatvec
    call(h, zbc.to_colmajor(A.astype(np.complex64)), B, zbc.AUTO if prec is None else prec)
    zbc.zbc_product_status(h)
    return zbc.from_colmajor(B)


@pytest.mark.parametrize("r", [(8, 70, 6), (8, 6, 70)])
def test_ranks_above_the_basis_keep_the_other_forms(r):
    g, tens = _shared((12, 80, 80), 20, (12, 80, 80), r)
    h = zbc.zbc_create_from_host(g, 3, tens)
    for tuned in (False, True):
        if tuned:
            zbc.zbc_tune(h, 9)
        for p in (2, 9):
            X = _c64(inputs.cn01((20, p), seed=1))
            Phi = _c64(inputs.cn01((3 * g.nv, p), seed=2))
            assert _rel(_run(h, g, X, True), products.matvec(tens, g.shape, X)) < RTOL
            assert _rel(_run(h, g, Phi, False), products.rmatvec(tens, g.shape, Phi)) < RTOL


def test_rank_above_the_product_kernels_is_refused():
    g, tens = _shared((80, 12, 12), 4, (80, 12, 12), (70, 6, 6))
    h = zbc.zbc_create_from_host(g, 3, tens)
    for call in (lambda: _run(h, g, np.ones((4, 2)), True), lambda: _run(h, g, np.ones((3 * g.nv, 2)), False),
                 lambda: zbc.zbc_tune(h, 2)):
        with pytest.raises(zbc.ZbcError) as e:
            call()
        assert e.value.status == zbc.ZBC_EINVAL


@pytest.mark.parametrize("form,sizes", [("fp32", (17, 32)), ("auto", (5, 17, 33, 64, 66))])
def test_a_smaller_product_keeps_the_buffers_of_a_larger_one(form, sizes):
    """A captured graph holds the buffers of its call: no call of fewer right-hand sides moves them."""
    prec = zbc.FP32_SIMT if form == "fp32" else zbc.AUTO
    g, tens = _shared((24, 24, 24), 130, (12, 12, 12), (6, 6, 6))
    for first in sizes:
        h = zbc.zbc_create_from_host(g, 3, tens)
        for fwd in (True, False):
            _run(h, g, np.ones((130 if fwd else 3 * g.nv, first)), fwd, prec)
        work = h.device_bytes()["work"]
        for p in range(first, 0, -1):
            for fwd in (True, False):
                _run(h, g, np.ones((130 if fwd else 3 * g.nv, p)), fwd, prec)
            assert h.device_bytes()["work"] == work, (first, p)


def _filled(leave):
    """All but `leave` bytes of the free device memory."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("first", ["matvec", "rmatvec", "tune"])
def test_products_without_room_for_the_reduced_cores(first):
    """Room for the decompression cache, but not for it and the joint form's cores (0.5 GB each)."""
    g, tens = _shared((96, 96, 96), 256, (44, 44, 44), (8, 8, 8))
    h, free = (zbc.zbc_create_from_host(g, 3, tens) for _ in range(2))
    X = zbc.to_colmajor(inputs.cn01((256, 2), seed=1).astype(np.complex64))
    Phi = zbc.to_colmajor(inputs.cn01((3 * g.nv, 2), seed=2).astype(np.complex64))
    Y, Psi = zbc.colmajor(3 * g.nv, 2, torch.complex64), zbc.colmajor(256, 2, torch.complex64)
    zbc.zbc_matvec(free, X, Y, zbc.FP32_SIMT)
    zbc.zbc_rmatvec(free, Phi, Psi, zbc.FP32_SIMT)
    want = Y.clone(), Psi.clone()
    W = free.device_bytes()["caches"]
    del free
    fill = _filled(W + (400 << 20))
    try:
        if first == "matvec":
            zbc.zbc_matvec(h, X, Y, zbc.AUTO)
        elif first == "rmatvec":
            zbc.zbc_rmatvec(h, Phi, Psi, zbc.AUTO)
        else:
            zbc.zbc_tune(h, 2)
        for prec in (zbc.AUTO, zbc.FP32_SIMT):
            zbc.zbc_matvec(h, X, Y, prec)
            zbc.zbc_rmatvec(h, Phi, Psi, prec)
            zbc.zbc_product_status(h)
            for got, ref in ((Y, want[0]), (Psi, want[1])):
                assert torch.linalg.norm(got - ref) < RTOL * torch.linalg.norm(ref)
        assert torch.equal(Y, want[0])
    finally:
        del fill
        torch.cuda.empty_cache()
    zbc.zbc_tune(h, 2)  # with the memory back, the joint form gets its cores
    assert h.device_bytes()["caches"] > W + (400 << 20)


def test_products_without_room_for_the_joint_workspace():
    g, tens = _shared((96, 96, 96), 256, (44, 44, 44), (8, 8, 8))
    h = zbc.zbc_create_from_host(g, 3, tens)
    A = [zbc.to_colmajor(inputs.cn01((256, p), seed=p).astype(np.complex64)) for p in (1, 2)]
    Y = [zbc.colmajor(3 * g.nv, p, torch.complex64) for p in (1, 2, 2)]
    zbc.zbc_matvec(h, A[1], Y[2], zbc.FP32_SIMT)
    zbc.zbc_matvec(h, A[0], Y[0], zbc.AUTO)  # the basis, and a workspace for one right-hand side
    fill = _filled(6 << 20)
    try:
        zbc.zbc_matvec(h, A[1], Y[1], zbc.AUTO)
        zbc.zbc_product_status(h)
        assert torch.equal(Y[1], Y[2])
    finally:
        del fill
        torch.cuda.empty_cache()


@pytest.mark.parametrize("p", [2, 6, 17])
@pytest.mark.parametrize("scale,norm", [(1e-36, 1.0), (1.0, 1e-8), (1e35, 1e-8)])
def test_scaled_vectors(p, scale, norm):
    g, tens = _shared((40, 36, 20), 48, (12, 11, 10), (6, 5, 4), norm=norm)
    h = zbc.zbc_create_from_host(g, 3, tens)
    X = _c64(inputs.cn01((48, p), seed=1) * scale)
    Phi = _c64(inputs.cn01((3 * g.nv, p), seed=2) * scale)
    assert _rel(_run(h, g, X, True), products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(_run(h, g, Phi, False), products.rmatvec(tens, g.shape, Phi)) < RTOL


@pytest.mark.parametrize("p", [2, 6, 17])
def test_small_column_against_a_small_entry(p):
    """A column of 1e-18 times the others' norm, alone in X with an entry of 1e-21."""
    g, tens = _shared((40, 36, 20), 48, (12, 11, 10), (6, 5, 4), norm=1e8)
    tens[7] = [(_c64(G * 1e-18), U) for G, U in tens[7]]
    h = zbc.zbc_create_from_host(g, 3, tens)
    X = np.zeros((48, p), np.complex128)
    X[7] = _c64(inputs.cn01((p,), seed=1) * 1e-21)
    Phi = _c64(inputs.cn01((3 * g.nv, p), seed=2))
    assert _rel(_run(h, g, X, True), products.matvec(tens, g.shape, X)) < RTOL
    Psi, ref = _run(h, g, Phi, False), products.rmatvec(tens, g.shape, Phi)
    assert _rel(Psi, ref) < RTOL and _rel(Psi[7:8].T, ref[7:8].T) < RTOL


@pytest.mark.parametrize("p", [2, 6, 17])
def test_nan_is_reported_and_stays_in_its_column(p):
    g, tens = _shared((40, 36, 20), 48, (12, 11, 10), (6, 5, 4))
    h = zbc.zbc_create_from_host(g, 3, tens)
    for fwd in (True, False):
        A = zbc.colmajor(48 if fwd else 3 * g.nv, p, torch.complex64)
        B = zbc.colmajor(3 * g.nv if fwd else 48, p, torch.complex64)
        A.fill_(1.0)
        A[1, 11] = float("nan")
        (zbc.zbc_matvec if fwd else zbc.zbc_rmatvec)(h, A, B, zbc.AUTO)
        with pytest.raises(zbc.ZbcError) as e:
            zbc.zbc_product_status(h)
        assert e.value.status == zbc.ZBC_ENAN
        ok = torch.isfinite(torch.view_as_real(B)).flatten(1)
        assert not ok[1].any() and ok[0].all() and ok[2:].all()


@pytest.mark.parametrize("p", [2, 16])
def test_accuracy(p):
    """Factors in exact common bases, so that only the arithmetic errs.  Its FP32 chains have at most 64
    terms, sqrt(64 / 2) 2^-24 / sqrt(3) = 2e-7 of a sum of random terms, in four passes of which each adds
    less than that: 4e-7, and 1e-7 for operands in FP32.  Truncating accumulators would shift the mean by 4.3e-8
    times half the sums they round, 1e-6 here; what is put back for them is a multiple of 2^-23 per pass."""
    g, tens = _shared((96, 90, 64), 96, (56, 56, 48), (16, 16, 16))
    h = zbc.zbc_create_from_host(g, 3, tens)
    X = _c64(inputs.cn01((96, p), seed=1))
    Phi = _c64(inputs.cn01((3 * g.nv, p), seed=2))
    for A, ref, fwd in ((X, products.matvec, True), (Phi, products.rmatvec, False)):
        got, ref = _run(h, g, A, fwd).astype(np.complex128), ref(tens, g.shape, A)
        assert _rel(got, ref) < 5e-7
        assert abs(np.vdot(ref, got).real / np.linalg.norm(ref) ** 2 - 1) < 1.5e-7


@pytest.mark.parametrize("p", [2, 9, 40])
@pytest.mark.parametrize("fwd", [True, False])
def test_a_wait_that_gives_up_is_reported_and_the_next_product_is_right(fwd, p):
    g, tens = _shared((300, 36, 20), 150, (12, 11, 10), (6, 5, 4))  # several blocks of i1, tiles of rows
    h = zbc.zbc_create_from_host(g, 3, tens)
    A = _c64(inputs.cn01((150 if fwd else 3 * g.nv, p), seed=1))
    ref = (products.matvec if fwd else products.rmatvec)(tens, g.shape, A)
    assert _rel(_run(h, g, A, fwd), ref) < RTOL
    zbc.zbc_test_wait_limit(h, 0)
    with pytest.raises(zbc.ZbcError) as e:
        _run(h, g, A, fwd)
    assert e.value.status == zbc.ZBC_ETIMEOUT
    assert _rel(_run(h, g, A, fwd), ref) < RTOL  # the limit was for one product, and the word is clear


def test_tuning_keeps_what_an_untuned_class_runs():
    """A graph of an untuned class survives the tuning of another one, whichever form that selects."""
    g, tens = _shared((24, 24, 24), 40, (10, 10, 10), (6, 6, 6))
    h = zbc.zbc_create_from_host(g, 3, tens)
    A = zbc.to_colmajor(inputs.cn01((40, 2), seed=1).astype(np.complex64))
    Y, Z = (zbc.colmajor(3 * g.nv, 2, torch.complex64) for _ in range(2))
    zbc.zbc_matvec(h, A, Y, zbc.AUTO)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        zbc.zbc_matvec(h, A, Z, zbc.AUTO)
    held = h.device_bytes()["caches"]
    for p in (1, 12, 64):
        zbc.zbc_tune(h, p)
        assert h.device_bytes()["caches"] >= held, p
    graph.replay()
    torch.cuda.synchronize()
    zbc.zbc_product_status(h)
    assert torch.equal(Y, Z)


def test_untuned_class_after_tuning_without_the_joint_form():
    """Tuned on its own, the handle drops the joint form if it lost, and an untuned class leaves it so."""
    g, tens = _shared((24, 24, 24), 40, (10, 10, 10), (6, 6, 6))
    h = zbc.zbc_create_from_host(g, 3, tens)
    zbc.zbc_tune(h, 1)
    held = h.device_bytes()["caches"]
    X = _c64(inputs.cn01((40, 12), seed=1))
    assert _rel(_run(h, g, X, True), products.matvec(tens, g.shape, X)) < RTOL
    assert h.device_bytes()["caches"] == held


# the adjoint's stages of i2: of 64 where they hold no more padding than stages of 32, cut at the rows where they
# hold more, several a tile, several tiles
@pytest.mark.parametrize("n2", [31, 33, 64, 65, 67, 81, 96, 100, 128, 129, 159, 187, 193, 256])
@pytest.mark.parametrize("n1,r", [(24, 7), (25, 20)])
def test_stages_of_the_adjoint_planes(n1, n2, r):
    g, tens = _shared((n1, n2, 10), 40, (r, r, 8), (5, 5, 4))
    h = zbc.zbc_create_from_host(g, 3, tens)
    Phi = _c64(inputs.cn01((3 * g.nv, 3), seed=2))
    assert _rel(_run(h, g, Phi, False), products.rmatvec(tens, g.shape, Phi)) < RTOL
