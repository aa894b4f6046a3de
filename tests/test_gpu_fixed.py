"""FP64 products in fixed point (PolI64 in csrc/common.cuh) at the edges of the
ring kernel's thread layouts, ragged segments, scaled, zero and non-finite
states, and the blocks that keep the FP64 kernel."""
import numpy as np
import pytest
import torch

import oracle
from paper_1201_6062_gb300 import inputs

pytestmark = pytest.mark.gpu


def reference(U, c, lmax, n, gauge="length"):
    """D c and, per amplitude, the bound n (max|u| max|x|) of its products, in extended precision."""
    x = c.reshape(lmax + 1, n).astype(np.clongdouble)
    y, b = np.zeros_like(x), np.zeros((lmax + 1, n))
    for l in range(lmax):
        u = U[l].astype(np.longdouble)
        s = 1j if gauge == "velocity" else 1.0
        y[l] += s * (u @ x[l + 1].real + 1j * (u @ x[l + 1].imag))
        y[l + 1] += np.conj(s) * (u.T @ x[l].real + 1j * (u.T @ x[l].imag))
        um = np.abs(U[l]).max(initial=0.0)
        amp = np.maximum(np.abs(c.real), np.abs(c.imag)).reshape(lmax + 1, n).max(1)
        b[l] += n * um * amp[l + 1]
        b[l + 1] += n * um * amp[l]
    return y.reshape(-1), b.reshape(-1)


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


# Three roundings of 2^-58 of max|u| max|x| per product at most (u and x to 58 bits of maxima rounded up
# to a power of two, the product of the low parts), four FP64 roundings of the result's sums.
def check(y, ref, bound):
    err = np.abs(y - ref).astype(np.float64)
    assert np.all(err <= 4 * 2.0 ** -58 * bound + 4 * 2.0 ** -53 * np.abs(ref).astype(np.float64))
    # and in the 2-norm no further off than sums rounded at every step
    assert np.linalg.norm(err) <= 5e-16 * np.linalg.norm(ref.astype(np.complex128))


@pytest.mark.parametrize("lmax,n", [(2, 65), (1, 128), (1, 255), (3, 257), (1, 512), (1, 513), (1, 768), (1, 769),
                                    (1, 1025), (1, 1153), (1, 1537), (1, 2047), (1, 2048), (1, 2050)])
def test_products_at_layout_edges(tdse_lib, lmax, n):
    U, c = random(lmax, n, n)
    check(product(tdse_lib, U, c, lmax, n), *reference(U, c, lmax, n))


@pytest.mark.parametrize("scale", [1e-200, 1e-3, 1e180])
def test_the_scale_of_blocks_and_states_does_not_matter(tdse_lib, scale):
    lmax, n = 3, 150
    U, c = random(lmax, n, 2)
    U *= np.array([1e-20, 1.0, 1e30])[:, None, None]
    c = c.reshape(lmax + 1, n) * np.array([1.0, 1e-12, 0.0, 1e5])[:, None]
    c = (c * scale).reshape(-1)
    for gauge in ("length", "velocity"):
        y = product(tdse_lib, U, c, lmax, n, gauge).reshape(lmax + 1, n)
        ref, b = (v.reshape(lmax + 1, n) for v in reference(U, c, lmax, n, gauge))
        for l in range(lmax + 1):
            assert np.all(np.abs(y[l] - ref[l]).astype(np.float64) <= 4 * 2.0 ** -58 * b[l] + 4 * 2.0 ** -53 * np.abs(ref[l]).astype(np.float64)), l


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


@pytest.mark.parametrize("what", ["rows", "columns", "nan", "zero rows"])
def test_blocks_the_fixed_point_would_not_serve(tdse_lib, what):
    lmax, n = 2, 130
    U, c = random(lmax, n, 4)
    if what == "rows":
        U[0] *= np.exp(-np.arange(n) / 4.0)[:, None]
    elif what == "columns":
        U[1] *= np.exp(-np.arange(n) / 4.0)[None, :]
    elif what == "nan":
        U[0, 3, 5] = np.nan
    else:
        U[0, ::3] = 0.0
    y = product(tdse_lib, U, c, lmax, n)
    if what == "nan":
        k = np.flatnonzero(~np.isfinite(y.real))
        assert list(k) == [3, n + 5]
        return
    ref, _ = reference(U, c, lmax, n)
    # each output relative to the sum of its own terms' magnitudes
    x = np.abs(c).reshape(lmax + 1, n)
    own = np.zeros((lmax + 1, n))
    for l in range(lmax):
        own[l] += np.abs(U[l]) @ x[l + 1]
        own[l + 1] += np.abs(U[l]).T @ x[l]
    assert np.all(np.abs(y - ref).astype(np.float64) <= 2.0 ** -50 * own.reshape(-1))


def test_without_room_for_the_copy_the_fp64_kernel_serves(tdse_lib):
    lmax, n, dt, steps = 3, 200, 0.02, 5
    E, U = inputs.energies(lmax, n), inputs.dipoles(lmax, n, 5)
    F = np.full(steps + 1, 0.1)
    c0 = inputs.random_state((lmax + 1) * n, 1)
    base = tdse_lib.device_memory_in_use()
    H = tdse_lib.Hamiltonian(E, U, lmax, n, "fp64")
    full = tdse_lib.device_memory_in_use() - base
    H.close()
    copy = lmax * n * n * 8
    tdse_lib.set_device_memory_limit(base + full - copy // 2)
    try:
        H = tdse_lib.Hamiltonian(E, U, lmax, n, "fp64")
    finally:
        tdse_lib.set_device_memory_limit(0)
    assert tdse_lib.device_memory_in_use() - base < full - copy // 2
    H2 = tdse_lib.Hamiltonian(E, U, lmax, n, "fp64")
    ref, _ = oracle.rk4(lmax, n, E, U, c0, F, dt, steps)
    # alone, and together with a member that has the copy
    for h in (H, H2):
        c = torch.from_numpy(c0.copy()).cuda()
        h.propagate(c, torch.from_numpy(F).cuda(), dt, steps)
        assert np.linalg.norm(c.cpu().numpy() - ref) < 1e-12
    for persistent in (False, True):
        g = tdse_lib.Group([H, H2])
        g.set_persistent(persistent)
        cs = [torch.from_numpy(c0.copy()).cuda() for _ in range(2)]
        g.propagate(cs, [torch.from_numpy(F).cuda()] * 2, dt, steps)
        g.sync()
        g.close()
        for c in cs:
            assert np.linalg.norm(c.cpu().numpy() - ref) < 1e-12
    H.close()
    H2.close()


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
