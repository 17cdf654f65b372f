"""The binding's amplitude layouts: flat (re, im) pairs against the element-wise
form, over types, orders and strides (no GPU)."""
import numpy as np
import pytest

from paper_1807_00699_gb300.gda import _amplitudes, _interleave

X = np.random.default_rng(0).normal(size=(4, 6)) + 1j * np.random.default_rng(1).normal(size=(4, 6))


@pytest.mark.parametrize("x", [X, X.astype(np.complex64), X[:, ::-1], X[::2], np.asfortranarray(X), X.real, X.T.T],
                         ids=["c128", "c64", "reversed", "strided", "fortran", "real", "view"])
def test_interleave(x):
    assert np.array_equal(_interleave(x, True), np.stack([x.real, x.imag], axis=-1).astype(np.float32).ravel())
    assert np.array_equal(_interleave(x.real, False), np.ascontiguousarray(x.real, dtype=np.float32).ravel())


@pytest.mark.parametrize("R,N", [(1, 1), (3, 5), (2, 8)])
def test_amplitudes(R, N):
    flat = np.random.default_rng(2).normal(size=2 * R * N).astype(np.float32)
    p = flat.reshape(R, N, 2)
    got = _amplitudes(flat.copy(), R, N, 2)
    assert got.dtype == np.complex64 and np.array_equal(got, p[..., 0] + 1j * p[..., 1])
    got[0, 0] = 0  # the caller's own array
    assert np.array_equal(_amplitudes(flat[:R * N], R, N, 1), flat[:R * N].reshape(R, N))
