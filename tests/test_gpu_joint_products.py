"""The joint-subspace form of both products, which ZBC_AUTO runs on an untuned handle whose columns'
factors share a small basis: against the FP64 oracle at the sizes where its kernels change shape
(ragged grids and tiles, passes and batches of right-hand sides, few and many columns, ACA storage,
q = 12, masked voxels), its status word, stream capture, and the handles that must not take it."""
import numpy as np
import pytest

from oracle import greens, products, tucker
from paper_2103_06393_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()
from paper_2103_06393_gb300 import zbc  # noqa: E402

# FP32 sums of at most a few thousand terms of the same scale: sqrt(4000) 2^-24 = 4e-6, and the
# basis adds at most sqrt(3) 1e-7
RTOL = 5e-6
FWD, ADJ = 3, 4  # kernels of the joint form for up to 64 right-hand sides


def _tensors(n, m, name="large", tol=1e-6, q=3, h=None):
    w = inputs.scaled_workload(name, n, m=m)
    g, s = w.grid, w.segments
    if h is not None:
        g = inputs.Grid(*n, h)
    Z = greens.assemble_columns(g.shape, g.h, s.centre, s.tangent, s.length, w.freq_hz, np.arange(s.m),
                                mask_radius=g.mask_radius, mask_box=g.mask_box)
    if q == 12:  # twelve row blocks of the same kind of field
        Z = np.concatenate([Z * f for f in (1.0, 0.3, -0.2, 0.1j)], axis=0)
    tens = tucker.compress_columns(Z, g.shape, q, tol)
    return g, [[(t[0].astype(np.complex64).astype(np.complex128),
                 [U.astype(np.complex64).astype(np.complex128) for U in t[1]]) for t in tj] for tj in tens]


def _rel(a, b):
    return float(np.max(np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)))


def _both(h, g, m, p, q=3, seed=0):
    X = inputs.cn01((m, p), seed=seed).astype(np.complex64)
    Phi = inputs.cn01((q * g.nv, p), seed=seed + 1).astype(np.complex64)
    Y = zbc.colmajor(q * g.nv, p, torch.complex64)
    Psi = zbc.colmajor(m, p, torch.complex64)
    Y.fill_(float("nan"))
    Psi.fill_(float("nan"))
    Xd, Pd = zbc.to_colmajor(X), zbc.to_colmajor(Phi)
    zbc.zbc_matvec(h, Xd, Y, zbc.AUTO)
    zbc.zbc_rmatvec(h, Pd, Psi, zbc.AUTO)
    launches = []
    for call in (lambda: zbc.zbc_matvec(h, Xd, Y, zbc.AUTO), lambda: zbc.zbc_rmatvec(h, Pd, Psi, zbc.AUTO)):
        l0 = zbc.kernel_launches()
        call()
        launches.append(zbc.kernel_launches() - l0)
    zbc.zbc_product_status(h)
    return X, Phi, zbc.from_colmajor(Y), zbc.from_colmajor(Psi), launches


# n1 around one and several i1 blocks of 32 NI rows; n2 and n3 off their tiles of 32 / 64 and 16
@pytest.mark.parametrize("n,m,p", [((40, 33, 17), 64, 1), ((33, 40, 65), 33, 2), ((64, 31, 16), 40, 3),
                                   ((129, 20, 24), 65, 5), ((100, 66, 12), 32, 9), ((24, 24, 40), 130, 17),
                                   ((161, 12, 20), 40, 16), ((40, 36, 20), 36, 70)])
def test_matches_oracle(n, m, p):
    g, tens = _tensors(n, m)
    h = zbc.zbc_create_from_host(g, 3, tens)
    X, Phi, Y, Psi, launches = _both(h, g, m, p)
    batches = -(-p // 64)
    assert launches == [FWD * batches, ADJ * batches]
    assert _rel(Y, products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec(tens, g.shape, Phi)) < RTOL


@pytest.mark.parametrize("name,n,m,p,h", [("large", (700, 12, 10), 32, 5, 4e-4),      # several groups of i1 blocks
                                          ("large", (20, 260, 12), 40, 6, 1e-3),      # several tiles of i2
                                          ("precision", (96, 100, 24), 64, 33, 2e-3)])  # the largest bases
def test_matches_oracle_at_the_plane_kernels_edges(name, n, m, p, h):
    g, tens = _tensors(n, m, name=name, h=h)
    hd = zbc.zbc_create_from_host(g, 3, tens)
    X, Phi, Y, Psi, launches = _both(hd, g, m, p)
    assert launches == [FWD, ADJ]
    assert _rel(Y, products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec(tens, g.shape, Phi)) < RTOL


def test_unaligned_vectors():
    """Columns that start off 16 bytes, and odd leading dimensions, on an even grid."""
    g, tens = _tensors((40, 36, 20), 40)
    h = zbc.zbc_create_from_host(g, 3, tens)
    X, Phi, Y, Psi, _ = _both(h, g, 40, 6)
    rows = 3 * g.nv
    buf = torch.zeros((6, rows + 3), dtype=torch.complex64, device="cuda")
    out = torch.zeros((6, 43), dtype=torch.complex64, device="cuda")
    P, O = buf[:, 1:1 + rows], out[:, 1:41]
    P.copy_(zbc.to_colmajor(Phi))
    zbc.zbc_rmatvec(h, P, O, zbc.AUTO)
    Xb = torch.zeros((6, 43), dtype=torch.complex64, device="cuda")
    Xb[:, 1:41].copy_(zbc.to_colmajor(X))
    P.fill_(float("nan"))
    zbc.zbc_matvec(h, Xb[:, 1:41], P, zbc.AUTO)
    zbc.zbc_product_status(h)
    assert _rel(zbc.from_colmajor(O), products.rmatvec(tens, g.shape, Phi)) < RTOL
    assert _rel(zbc.from_colmajor(P), products.matvec(tens, g.shape, X)) < RTOL
    assert not buf[:, 0].any() and not buf[:, 1 + rows:].any()


def test_masked_grid_keeps_exact_zeros():
    g, tens = _tensors((160, 24, 20), 40, name="batching")
    keep = np.abs(g.axis(0)) <= g.mask_box
    assert 0 < keep.sum() < g.n1
    for tj in tens:
        for _, U in tj:
            U[0][~keep] = 0  # the oracle's SVD leaves rounding there; the GPU compressor exact zeros
    h = zbc.zbc_create_from_host(g, 3, tens)
    X, Phi, Y, Psi, launches = _both(h, g, 40, 4)
    assert launches == [FWD, ADJ]
    assert _rel(Y, products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec(tens, g.shape, Phi)) < RTOL
    assert not Y.reshape(3, g.n3, g.n2, g.n1, 4)[..., ~keep, :].any()


def test_twelve_row_blocks():
    g, tens = _tensors((36, 30, 20), 40, q=12)
    h = zbc.zbc_create_from_host(g, 12, tens)
    X, Phi, Y, Psi, launches = _both(h, g, 40, 3, q=12)
    assert launches == [FWD, ADJ]
    assert _rel(Y, products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec(tens, g.shape, Phi)) < RTOL


def test_aca_storage():
    g, tens = _tensors((40, 36, 20), 40)
    V = inputs.cn01((90, 40), seed=5).astype(np.complex64)
    h = zbc.zbc_create_from_host(g, 3, tens, V)
    X, Phi, Y, Psi, launches = _both(h, g, 90, 3)
    assert launches == [FWD + 1, ADJ + 1]
    Vd = V.astype(np.complex128)
    assert _rel(Y, products.matvec_aca(tens, Vd, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec_aca(tens, Vd, g.shape, Phi)) < RTOL


def test_columns_of_very_different_norm():
    """The basis bounds each tensor's error by its own norm: a column 1e-12 of the others' size,
    alone in X, comes out as exactly as the others."""
    g, tens = _tensors((40, 36, 20), 40)
    tens[7] = [(G * 1e-12, U) for G, U in tens[7]]
    h = zbc.zbc_create_from_host(g, 3, tens)
    X = np.zeros((40, 2), np.complex64)
    X[7, 0] = 1.0
    X[8, 1] = 1.0
    Y = zbc.colmajor(3 * g.nv, 2, torch.complex64)
    zbc.zbc_matvec(h, zbc.to_colmajor(X), Y, zbc.AUTO)
    assert _rel(zbc.from_colmajor(Y), products.matvec(tens, g.shape, X)) < RTOL


@pytest.mark.parametrize("scale", [1e-25, 1e25])
def test_scaled_right_hand_sides(scale):
    g, tens = _tensors((40, 36, 20), 40)
    h = zbc.zbc_create_from_host(g, 3, tens)
    X, _, Y, Psi, _ = _both(h, g, 40, 3)
    Xs = zbc.to_colmajor((X * scale).astype(np.complex64))
    Ys = zbc.colmajor(3 * g.nv, 3, torch.complex64)
    zbc.zbc_matvec(h, Xs, Ys, zbc.AUTO)
    ref = products.matvec(tens, g.shape, zbc.from_colmajor(Xs).astype(np.complex128))
    assert _rel(zbc.from_colmajor(Ys).astype(np.complex128), ref) < RTOL


def test_nan_input_is_reported():
    g, tens = _tensors((40, 36, 20), 40)
    h = zbc.zbc_create_from_host(g, 3, tens)
    _both(h, g, 40, 2)
    for fwd in (True, False):
        A = zbc.colmajor(40 if fwd else 3 * g.nv, 2, torch.complex64)
        A.fill_(1.0)
        A[1, 11] = float("nan")
        B = zbc.colmajor(3 * g.nv if fwd else 40, 2, torch.complex64)
        (zbc.zbc_matvec if fwd else zbc.zbc_rmatvec)(h, A, B, zbc.AUTO)
        with pytest.raises(zbc.ZbcError) as e:
            zbc.zbc_product_status(h)
        assert e.value.status == zbc.ZBC_ENAN
        b = torch.view_as_real(B)
        assert torch.isfinite(b[0]).all() and not torch.isfinite(b[1]).any()


def test_unrelated_factors_keep_the_other_forms():
    """Random factors span everything: AUTO runs what it ran without a joint basis, bit for bit."""
    rng = np.random.default_rng(3)
    g = inputs.Grid(72, 70, 66, 0.001)

    def tensor():
        U = [np.linalg.qr(rng.normal(size=(n, 4)) + 1j * rng.normal(size=(n, 4)))[0] for n in g.shape]
        return rng.normal(size=(4, 4, 4)) + 1j * rng.normal(size=(4, 4, 4)), U

    h = zbc.zbc_create_from_host(g, 3, [[tensor() for _ in range(3)] for _ in range(40)])
    for p, form in ((2, zbc.FP32_SIMT), (9, zbc.BF16X3)):
        X = zbc.to_colmajor(inputs.cn01((40, p), seed=1).astype(np.complex64))
        Y = [zbc.colmajor(3 * g.nv, p, torch.complex64) for _ in range(2)]
        zbc.zbc_matvec(h, X, Y[0], zbc.AUTO)
        zbc.zbc_matvec(h, X, Y[1], form)
        assert torch.equal(Y[0], Y[1])


def test_append_builds_a_new_basis():
    w = inputs.scaled_workload("large", (40, 36, 20), m=48)
    g, s = w.grid, w.segments
    Z = greens.assemble_columns(g.shape, g.h, s.centre, s.tangent, s.length, w.freq_hz, np.arange(s.m))
    h, _ = zbc.tucker_compress(zbc.to_colmajor(Z[:, :24], np.complex128), g, 1e-6)
    _both(h, g, 24, 3)
    h, _ = zbc.tucker_compress(zbc.to_colmajor(Z[:, 24:], np.complex128), g, 1e-6, append_to=h)
    X, Phi, Y, Psi, _ = _both(h, g, 48, 3)
    tens, _ = h.tensors()
    assert _rel(Y, products.matvec(tens, g.shape, X)) < RTOL
    assert _rel(Psi, products.rmatvec(tens, g.shape, Phi)) < RTOL


def test_capture_without_a_basis_runs_the_form_it_ran():
    """A capture on a handle that has only seen explicit calls allocates nothing and replays them."""
    g, tens = _tensors((40, 36, 20), 40)
    h = zbc.zbc_create_from_host(g, 3, tens)
    X = zbc.to_colmajor(inputs.cn01((40, 4), seed=1).astype(np.complex64))
    Y, Z = (zbc.colmajor(3 * g.nv, 4, torch.complex64) for _ in range(2))
    zbc.zbc_matvec(h, X, Y, zbc.FP32_SIMT)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        zbc.zbc_matvec(h, X, Z, zbc.AUTO)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, Z)


@pytest.mark.parametrize("form", ["auto", "fp32"])
def test_graph_of_one_product_survives_the_other(form):
    """A captured forward keeps its buffers when the adjoint runs for the first time afterwards."""
    g, tens = _tensors((40, 36, 20), 40)
    h = zbc.zbc_create_from_host(g, 3, tens)
    prec = zbc.AUTO if form == "auto" else zbc.FP32_SIMT
    X = zbc.to_colmajor(inputs.cn01((40, 6), seed=1).astype(np.complex64))
    Phi = zbc.to_colmajor(inputs.cn01((3 * g.nv, 6), seed=2).astype(np.complex64))
    Y, Z = (zbc.colmajor(3 * g.nv, 6, torch.complex64) for _ in range(2))
    Psi = zbc.colmajor(40, 6, torch.complex64)
    zbc.zbc_matvec(h, X, Y, prec)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        zbc.zbc_matvec(h, X, Z, prec)
    work = h.device_bytes()["work"]
    zbc.zbc_rmatvec(h, Phi, Psi, prec)
    assert h.device_bytes()["work"] > work  # the adjoint took buffers of its own
    graph.replay()
    torch.cuda.synchronize()
    zbc.zbc_product_status(h)
    assert torch.equal(Y, Z)
