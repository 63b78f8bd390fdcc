"""The eigensolver, Gram and sketch kernels of the compressors at the sizes where they change: the
largest matrix that stays in shared memory and the next one, the smallest, matrices of full
numerical range and of none, few and many tensors (split and whole Gram sums), and sketch widths on
both sides of a group of 8 -- against the FP64 oracle's HOSVD: equal ranks outside the window of near
ties, and an error within the tolerance."""
import numpy as np
import pytest

from oracle import tucker
from paper_2103_06393_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()
from paper_2103_06393_gb300 import zbc  # noqa: E402


def _decaying(n, rng, rate):
    """A tensor whose unfoldings' singular values fall by about `rate` from one to the next."""
    A = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    for d in range(3):
        Q = np.linalg.qr(rng.standard_normal((n[d], n[d])) + 1j * rng.standard_normal((n[d], n[d])))[0]
        A = tucker.mode_product(A, Q * rate ** np.arange(n[d]), d)
    return A


def _check(A, t, tol):
    _, _, info = tucker.hosvd(A, tol)
    for mode, U in enumerate(t[1]):
        if info["margin"][mode] > 1e-5:
            assert U.shape[1] == info["ranks"][mode], (mode, U.shape[1], info["ranks"], info["margin"])
        assert np.abs(U.conj().T @ U - np.eye(U.shape[1])).max() < 1e-6
    err = np.linalg.norm(tucker.reconstruct(*t) - A) / max(np.linalg.norm(A), 1e-300)
    assert err <= tol * (1 + 1e-6) + 3e-7


@pytest.mark.parametrize("n,rate,tol,m", [((116, 6, 4), 0.5, 1e-6, 2), ((118, 6, 4), 0.5, 1e-6, 2),
                                          ((8, 116, 10), 0.7, 1e-8, 2), ((2, 4, 6), 1.0, 1e-3, 3),
                                          ((24, 26, 28), 1.0, 1e-8, 2), ((30, 12, 64), 0.3, 1e-2, 60)])
def test_hosvd_of_decaying_tensors(n, rate, tol, m):
    rng = np.random.default_rng(7)
    tens = [_decaying(n, rng, rate) for _ in range(m)]
    cols = np.stack([A.reshape(-1, order="F") for A in tens], axis=1)
    h, st = zbc.tucker_compress(zbc.to_colmajor(cols), inputs.Grid(*n, 0.001), tol, q=1)
    got, _ = h.tensors()
    for A, t in zip(tens, got):
        _check(A, t[0], tol)
    assert st.max_rel_err <= tol * (1 + 1e-9)


def test_zero_and_rank_one_tensors():
    n = (12, 10, 8)
    rng = np.random.default_rng(3)
    one = np.einsum("a,b,c->abc", *[rng.standard_normal(k) + 1j * rng.standard_normal(k) for k in n])
    cols = np.stack([np.zeros(n).reshape(-1), one.reshape(-1, order="F")], axis=1)
    h, _ = zbc.tucker_compress(zbc.to_colmajor(cols, np.complex128), inputs.Grid(*n, 0.001), 1e-6, q=1)
    (zero,), (t,) = h.tensors()[0]
    assert zero[0].shape == t[0].shape == (1, 1, 1) and not zero[0].any()
    _check(one, t, 1e-6)


@pytest.mark.parametrize("width", [2, 8, 10, 24, 26, 40, 44, 48, 64])
def test_randomized_at_sketch_widths(width):
    n, tol = (70, 66, 68), 1e-5
    rng = np.random.default_rng(11)
    r = min(width, 12) if width > 2 else 2
    G = rng.standard_normal((r, r, r)) + 1j * rng.standard_normal((r, r, r))
    A = tucker.reconstruct(G, [np.linalg.qr(rng.standard_normal((k, r)) + 1j * rng.standard_normal((k, r)))[0] for k in n])
    grid = inputs.Grid(*n, 0.001)
    sk = [torch.from_numpy(np.ascontiguousarray(s.T)).cuda() for s in inputs.mode_sketches(grid, width, seed=2)]
    h, st = zbc.tucker_compress(zbc.to_colmajor(A.reshape(-1, 1, order="F")), grid, tol, q=1,
                                method=zbc.RANDOMIZED_FIXED, model=zbc.rank_model(sk, width, fixed_width=width))
    assert st.n_fallback == 0
    _check(A, h.tensors()[0][0][0], tol)
