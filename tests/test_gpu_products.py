"""FP64 products of the ring kernel: every component against the sum of its own
terms' magnitudes, at the edges of the thread layouts, over graded blocks and
states, and with non-finite amplitudes."""
import numpy as np
import pytest
import torch

import oracle
from paper_1201_6062_gb300 import inputs

pytestmark = pytest.mark.gpu


def reference(U, c, lmax, n, gauge="length"):
    """D c in extended precision and, per amplitude, the sum of its terms' magnitudes."""
    x = c.reshape(lmax + 1, n).astype(np.clongdouble)
    y, own = np.zeros_like(x), np.zeros((lmax + 1, n))
    for l in range(lmax):
        u = U[l].astype(np.longdouble)
        s = 1j if gauge == "velocity" else 1.0
        y[l] += s * (u @ x[l + 1].real + 1j * (u @ x[l + 1].imag))
        y[l + 1] += np.conj(s) * (u.T @ x[l].real + 1j * (u.T @ x[l].imag))
        own[l] += (np.abs(u) @ np.abs(x[l + 1])).astype(float)
        own[l + 1] += (np.abs(u).T @ np.abs(x[l])).astype(float)
    return y.reshape(-1), own.reshape(-1)


def product(T, U, c, lmax, n, gauge="length"):
    H = T.Hamiltonian(np.zeros((lmax + 1) * n), U, lmax, n, "fp64")
    if gauge != "length":
        H.set_gauge(gauge)
    y = H.hmatvec(torch.from_numpy(c).cuda(), 1.0).cpu().numpy()
    H.close()
    return y


def random(lmax, n, seed):
    rng = np.random.default_rng(seed)
    U = rng.standard_normal((lmax, n, n)) / np.sqrt(n)
    c = rng.standard_normal((lmax + 1) * n) + 1j * rng.standard_normal((lmax + 1) * n)
    return U, c


# A sum of at most 2 n products in any order: n 2^-53 of its terms' magnitudes for each part, and the last addition.
def check(y, ref, own, n):
    err = np.abs(y - ref).astype(np.float64)
    assert np.all(err <= (2 * n + 2) * 2.0 ** -53 * own)


@pytest.mark.parametrize("lmax,n", [(2, 65), (1, 128), (1, 255), (3, 257), (1, 512), (1, 513), (1, 768), (1, 769),
                                    (1, 1025), (1, 1153), (1, 1537), (1, 2047), (1, 2048), (1, 2050)])
def test_products_at_layout_edges(tdse_lib, lmax, n):
    U, c = random(lmax, n, n)
    y, (ref, own) = product(tdse_lib, U, c, lmax, n), reference(U, c, lmax, n)
    check(y, ref, own, n)
    # and in the 2-norm, where roundings of n terms average out, a few units in the last place
    assert np.linalg.norm((y - ref).astype(np.complex128)) <= 5e-16 * np.linalg.norm(ref.astype(np.complex128))


@pytest.mark.parametrize("scale", [1e-200, 1e-3, 1e180])
def test_the_scale_of_blocks_and_states_does_not_matter(tdse_lib, scale):
    lmax, n = 3, 150
    U, c = random(lmax, n, 2)
    U *= np.array([1e-20, 1.0, 1e30])[:, None, None]
    c = c.reshape(lmax + 1, n) * np.array([1.0, 1e-12, 0.0, 1e5])[:, None]
    c = (c * scale).reshape(-1)
    for gauge in ("length", "velocity"):
        check(product(tdse_lib, U, c, lmax, n, gauge), *reference(U, c, lmax, n, gauge), n)


@pytest.mark.parametrize("what", ["rows", "columns", "dominant", "zero rows"])
def test_small_components_keep_their_digits(tdse_lib, what):
    """Blocks with rows or columns of very different size, and a bound state: one amplitude near 1 whose
    dipole elements fall off, the others at 1e-10."""
    lmax, n = 2, 301
    U, c = random(lmax, n, 4)
    if what == "rows":
        U[0] *= np.exp(-np.arange(n) / 4.0)[:, None]
    elif what == "columns":
        U[1] *= np.exp(-np.arange(n) / 4.0)[None, :]
    elif what == "dominant":
        fall = (1.0 + np.arange(n) / 5.0) ** -4
        U[:, :, 0] *= fall
        U[:, 0, :] *= fall
        c *= 1e-10
        c[::n] = 1.0
    else:
        U[0, ::3] = 0.0
    check(product(tdse_lib, U, c, lmax, n), *reference(U, c, lmax, n), n)


def test_a_non_finite_dipole_element_reaches_its_row_and_column_only(tdse_lib):
    lmax, n = 2, 130
    U, c = random(lmax, n, 4)
    U[0, 3, 5] = np.nan
    assert list(np.flatnonzero(~np.isfinite(product(tdse_lib, U, c, lmax, n).real))) == [3, n + 5]


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_amplitude_reaches_its_neighbours_only(tdse_lib, bad):
    lmax, n = 4, 100
    U, c = random(lmax, n, 3)
    clean = product(tdse_lib, U, c, lmax, n).reshape(lmax + 1, n)
    c[n + 7] = bad
    y = product(tdse_lib, U, c, lmax, n).reshape(lmax + 1, n)
    for l in (0, 2):
        assert not np.any(np.isfinite(y[l].real) & np.isfinite(y[l].imag))
    for l in (3, 4):
        assert np.array_equal(y[l], clean[l])


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-14), ("df32", 1e-11), ("fp32", 2e-6)])
@pytest.mark.parametrize("lmax,n", [(0, 70), (3, 40), (4, 301)])
def test_products_queued_without_a_wait(tdse_lib, lmax, n, prec, tol):
    """Products of different vectors queued one behind the other, and one
    recorded in a graph and replayed after another call: each reads the
    vectors it was called with.  Tolerances: the products' (fp64: 2^-53 times
    the square root of the terms of a sum)."""
    rng = np.random.default_rng(3)
    E, U = inputs.energies(lmax, n), rng.standard_normal((lmax, n, n)) / n ** 0.5
    H = tdse_lib.Hamiltonian(E, U, lmax, n, prec)
    X = rng.standard_normal((4, (lmax + 1) * n, 2)).view(np.complex128)[..., 0]
    x = torch.from_numpy(X.copy()).cuda()
    y = torch.zeros_like(x)
    for i in range(3):
        H.hmatvec(x[i], 0.3, y=y[i])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        H.hmatvec(x[3], 0.3, y=y[3])
    H.hmatvec(x[0], 0.3, y=y[0])
    g.replay()
    torch.cuda.synchronize()
    for i in range(4):
        ref = oracle.hmatvec(lmax, n, E, U, 0.3, X[i])
        assert np.linalg.norm(y[i].cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    H.close()


# 256, 128 and 64 amplitudes a block of the update (fewer blocks than SMs where it starts early), the last one ragged
@pytest.mark.parametrize("lmax,n", [(31, 653), (20, 487), (7, 301)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-14), ("df32", 1e-11), ("fp32", 2e-6)])
def test_update_blocks(tdse_lib, lmax, n, prec, tol):
    """One product and one RK4 step against plain FP64 arithmetic."""
    U, c = random(lmax, n, 7)
    c /= np.linalg.norm(c)
    E, dt, f = inputs.energies(lmax, n), 0.01, 0.05

    def hx(y):
        x = y.reshape(lmax + 1, n)
        d = np.zeros_like(x)
        d[:-1] += np.einsum("lij,lj->li", U, x[1:], optimize=True)
        d[1:] += np.einsum("lij,li->lj", U, x[:-1], optimize=True)
        return E * y + f * d.reshape(-1)

    H = tdse_lib.Hamiltonian(E, U, lmax, n, prec)
    x = torch.from_numpy(c.copy()).cuda()
    ref = hx(c)
    assert np.linalg.norm(H.hmatvec(x, f).cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    H.propagate(x, torch.full((2,), f, dtype=torch.float64, device="cuda"), dt, 1)
    k1 = -1j * ref
    k2 = -1j * hx(c + 0.5 * dt * k1)
    k3 = -1j * hx(c + 0.5 * dt * k2)
    ref = c + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 - 1j * hx(c + dt * k3))
    assert np.linalg.norm(x.cpu().numpy() - ref) <= tol
    H.close()
