"""The digit-sliced batched products (csrc/dig.cuh) at the edges of their
tiles: rows (128, 256), K rounds (64, 512), pulses per tile, end blocks, every
tile shape with several tiles a CTA, both gauges, bound, graded, zero and
non-finite states, and the paths and memory around them."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1201_6062_gb300 import inputs

pytestmark = pytest.mark.gpu

DIGITS = {"fp32": 7, "df32": 7, "fp64": 11}
# error of the products, relative 2-norm, that the FMA- and FP64-pipe kernels show at these sizes
NORM = {"fp32": 6e-7, "df32": 1e-11, "fp64": 2e-15}
# state arithmetic (float-float sums of the products: 2^-46 of the largest; FP64 elsewhere)
SUM = {"fp32": 2.0 ** -46, "df32": 2.0 ** -46, "fp64": 2.0 ** -50}


def product(T, prec, lmax, n, U, C, gauge="length"):
    """(1 - i D) c - c for every state: one Taylor term of order 1, E = 0, f = dt = 1."""
    B = len(C)
    H = T.Hamiltonian(np.zeros((lmax + 1) * n), U, lmax, n, prec)
    if gauge != "length":
        H.set_gauge(gauge)
    c = torch.from_numpy(C.copy()).cuda()
    H.propagate_batch(c, torch.ones(B, 2, dtype=torch.float64, device="cuda"), B, 1.0, 1, "taylor", order=1)
    H.sync()
    H.close()
    return c.cpu().numpy() - C


def draw(prec, lmax, n, B, seed, graded=False):
    rng = np.random.default_rng(seed)
    U = rng.standard_normal((lmax, n, n)) / np.sqrt(n)
    C = rng.standard_normal((B, (lmax + 1) * n)) + 1j * rng.standard_normal((B, (lmax + 1) * n))
    if graded:
        # every block and pulse on a scale of its own
        C *= np.exp(rng.uniform(-40, 10, (B, lmax + 1))).repeat(n, axis=1)
        U *= np.exp(rng.uniform(-20, 5, (lmax, n, 1)))
    if prec == "fp32":                            # FP32 contexts store U so; the digits are finer than its rounding
        U = U.astype(np.float32).astype(np.float64)
    return U, C


def check(prec, lmax, n, U, C, k, gauge="length"):
    S = DIGITS[prec]
    x = C.reshape(len(C), lmax + 1, n)
    k = k.reshape(x.shape)
    amax = np.maximum(np.abs(x.real).max(2), np.abs(x.imag).max(2))          # [B, L]
    for l in range(lmax + 1):
        ref = np.zeros((len(C), n), np.complex128)
        bound = np.zeros((len(C), n))
        if l < lmax:
            ref += (1j if gauge == "velocity" else 1.0) * (x[:, l + 1] @ U[l].T)
            bound += amax[:, l + 1, None] * np.abs(U[l]).max(1)[None]
        if l >= 1:
            ref += (-1j if gauge == "velocity" else 1.0) * (x[:, l - 1] @ U[l - 1])
            bound += amax[:, l - 1, None] * np.abs(U[l - 1]).max(0)[None]
        # digits left out: S - 1 pairs of weight S and half a unit of either operand's last
        # digit, against maxima rounded up to powers of two
        bound = n * bound * (S * 2.0 ** (4 - 8 * S) + SUM[prec]) + 2.0 ** -51 * (np.abs(x[:, l]) + np.abs(ref))
        err = np.abs(k[:, l] - -1j * ref)
        assert np.all(err <= 2 * bound), (l, float((err / np.maximum(bound, 1e-300)).max()))
        # relative to each pulse's block; the subtraction of c costs FP64 rounding of c
        nrm = np.linalg.norm(err, axis=1) - 2.0 ** -52 * np.linalg.norm(x[:, l], axis=1)
        assert np.all(nrm <= NORM[prec] * np.linalg.norm(ref, axis=1) + 1e-300), (l, nrm / np.linalg.norm(ref, axis=1))


SHAPES = [(1, 64, 1), (2, 65, 16), (1, 127, 17), (3, 128, 32), (1, 129, 33), (2, 200, 64), (1, 256, 65), (1, 257, 9),
          (2, 513, 9), (1, 640, 40)]


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
@pytest.mark.parametrize("lmax,n,B", SHAPES)
def test_products_at_tile_edges(tdse_lib, prec, lmax, n, B):
    U, C = draw(prec, lmax, n, B, 11 * n + B)
    C *= 1e3                                      # the products, not c, set the size of the result
    check(prec, lmax, n, U * 1024, C, product(tdse_lib, prec, lmax, n, U * 1024, C))


class Tile(ctypes.Structure):
    _fields_ = [("cg", ctypes.c_int), ("bn", ctypes.c_int)]


# (precisions, lmax, n, pulses): the tile (CTAs of 128 rows, pulse planes) the launch chooses, and more tiles than
# CTAs or pairs, so that a CTA hands its scratch tile, state slots and accumulators on from one tile to the next
WALKS = [(("fp32", "df32"), 90, 130, 16, (2, 32)), (("fp32", "df32"), 80, 130, 33, (2, 64)),
         (("fp32", "df32"), 20, 200, 300, (2, 128)), (("fp32", "df32"), 80, 64, 33, (1, 32)),
         (("fp32", "df32"), 40, 70, 130, (1, 64)), (("fp64",), 80, 130, 15, (2, 32)), (("fp64",), 80, 130, 33, (2, 64)),
         (("fp64",), 90, 64, 33, (1, 32)), (("fp64",), 50, 70, 100, (1, 64))]
WALKS = [(p,) + w[1:] for w in WALKS for p in w[0]]


def assert_walk(T, prec, lmax, n, B, tile):
    choose = T._lib._ZN4tdse8dig_tileEiiii
    choose.restype, choose.argtypes = Tile, [ctypes.c_int] * 4
    t = choose(DIGITS[prec], n, lmax, B)
    assert (t.cg, t.bn) == tile
    tiles = -(-n // (128 * t.cg)) * -(-2 * B // t.bn) * (lmax + 1)
    assert tiles > torch.cuda.get_device_properties(0).multi_processor_count // t.cg


@pytest.mark.parametrize("prec,lmax,n,B,tile", WALKS)
def test_several_tiles_a_cta(tdse_lib, prec, lmax, n, B, tile):
    assert_walk(tdse_lib, prec, lmax, n, B, tile)
    for gauge in ("length", "velocity"):
        U, C = draw(prec, lmax, n, B, n + B)
        C *= 1e3
        check(prec, lmax, n, U * 1024, C, product(tdse_lib, prec, lmax, n, U * 1024, C, gauge), gauge)


@pytest.mark.parametrize("prec,lmax,n,B,tile", WALKS)
@pytest.mark.parametrize("scheme", ["rk4", "taylor"])
def test_steps_over_several_tiles(tdse_lib, prec, lmax, n, B, tile, scheme):
    assert_walk(tdse_lib, prec, lmax, n, B, tile)
    dt, order = 0.01, 4 if scheme == "rk4" else 3
    U, C = draw(prec, lmax, n, B, n + B + 1)
    C /= np.linalg.norm(C, axis=1)[:, None]
    E = inputs.energies(lmax, n)
    F = 0.05 + 0.01 * np.random.default_rng(7).random((B, 2))
    H = tdse_lib.Hamiltonian(E, U, lmax, n, prec)
    c = torch.from_numpy(C.copy()).cuda()
    H.propagate_batch(c, torch.from_numpy(F).cuda(), B, dt, 1, scheme, order=order)
    H.sync()
    H.close()

    def g(y, f):
        x = y.reshape(B, lmax + 1, n)
        d = np.zeros_like(x)
        d[:, :-1] += np.einsum("lij,blj->bli", U, x[:, 1:], optimize=True)
        d[:, 1:] += np.einsum("lij,bli->blj", U, x[:, :-1], optimize=True)
        return -1j * (E * y + f[:, None] * d.reshape(B, -1))

    if scheme == "rk4":
        fm = 0.5 * (F[:, 0] + F[:, 1])
        k1 = g(C, F[:, 0])
        k2 = g(C + 0.5 * dt * k1, fm)
        k3 = g(C + 0.5 * dt * k2, fm)
        ref = C + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + g(C + dt * k3, F[:, 1]))
    else:
        term = ref = C
        for m in range(1, order + 1):
            term = dt / m * g(term, F[:, 0])
            ref = ref + term
    # a step changes the state by dt (|E| + f |D|) of it at most; products as in NORM, FP64 rounding of the rest
    err = np.linalg.norm(c.cpu().numpy() - ref, axis=1)
    assert np.all(err <= 4 * (dt * 0.06 * 4 * NORM[prec] + 8 * 2.0 ** -53)), err.max()


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
@pytest.mark.parametrize("gauge", ["length", "velocity"])
def test_graded_blocks_keep_their_own_scale(tdse_lib, prec, gauge):
    lmax, n, B = 3, 150, 20
    U, C = draw(prec, lmax, n, B, 5, graded=True)
    C[3] = 0.0
    C[4, n:2 * n] = 0.0
    k = product(tdse_lib, prec, lmax, n, U, C, gauge)
    assert not np.any(k[3])
    x = C.reshape(B, lmax + 1, n)
    S = DIGITS[prec]
    for l in range(lmax + 1):
        up, dn = np.zeros((B, n), np.complex128), np.zeros((B, n), np.complex128)
        bound = 2.0 ** -50 * np.abs(x[:, l])
        if l < lmax:
            up = (1j if gauge == "velocity" else 1.0) * (x[:, l + 1] @ U[l].T)
            bound = bound + (S * 2.0 ** (4 - 8 * S) + SUM[prec]) * n * np.abs(x[:, l + 1]).max(1)[:, None] * np.abs(U[l]).max(1)
        if l >= 1:
            dn = (-1j if gauge == "velocity" else 1.0) * (x[:, l - 1] @ U[l - 1])
            bound = bound + (S * 2.0 ** (4 - 8 * S) + SUM[prec]) * n * np.abs(x[:, l - 1]).max(1)[:, None] * np.abs(U[l - 1]).max(0)
        err = np.abs(k.reshape(x.shape)[:, l] - -1j * (up + dn))
        assert np.all(err <= 2 * (bound + 2.0 ** -50 * (np.abs(up) + np.abs(dn)))), l


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_pulse_stays_alone(tdse_lib, prec, bad):
    lmax, n, B = 2, 140, 18
    U, C = draw(prec, lmax, n, B, 6)
    clean = product(tdse_lib, prec, lmax, n, U, C)
    C2 = C.copy()
    C2[7, n + 5] = bad
    k = product(tdse_lib, prec, lmax, n, U, C2)
    assert not np.any(np.isfinite(k[7, :n].real) & np.isfinite(k[7, :n].imag))
    assert np.array_equal(np.delete(k, 7, 0), np.delete(clean, 7, 0))


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("df32", 1e-10), ("fp64", 1e-10)])
@pytest.mark.parametrize("scheme,order,sps", [("rk4", 4, 2), ("taylor", 3, 1)])
def test_windows_match_the_oracle(tdse_lib, prec, tol, scheme, order, sps):
    lmax, n, B, dt, steps = 3, 140, 19, 0.02, 12
    E, U = inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8)
    C = np.stack([inputs.random_state((lmax + 1) * n, b) for b in range(B)])
    F = np.stack([inputs.field_samples(0.1 + 0.01 * b, 0.5, dt, steps, sps, cycles=3, t0=3.0) for b in range(B)])
    H = tdse_lib.Hamiltonian(E, U, lmax, n, prec)
    c = torch.from_numpy(C.copy()).cuda()
    H.propagate_batch(c, torch.from_numpy(F).cuda(), B, dt, steps, scheme, order=order, samples_per_step=sps)
    H.sync()
    # again on the same context with fewer pulses (other digit planes and tiles)
    c2 = torch.from_numpy(C[:3].copy()).cuda()
    H.propagate_batch(c2, torch.from_numpy(F[:3].copy()).cuda(), 3, dt, steps, scheme, order=order, samples_per_step=sps)
    H.sync()
    H.close()
    for b in range(B):
        args = (lmax, n, E, U, C[b], F[b], dt, steps)
        ref, _ = oracle.rk4(*args, samples_per_step=sps) if scheme == "rk4" else oracle.taylor(*args, order, samples_per_step=sps)
        for got in ([c[b]] if b >= 3 else [c[b], c2[b]]):
            assert np.linalg.norm(got.cpu().numpy() - ref) < tol * np.linalg.norm(ref), b


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("df32", 1e-10), ("fp64", 1e-10)])
def test_without_room_for_digits_the_other_path_serves(tdse_lib, prec, tol):
    lmax, n, B, dt, steps = 2, 200, 12, 0.02, 3
    E, U = inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8)
    C = np.stack([inputs.random_state((lmax + 1) * n, b) for b in range(B)])
    F = np.full((B, steps + 1), 0.1)
    H = tdse_lib.Hamiltonian(E, U, lmax, n, prec)
    used = tdse_lib.device_memory_in_use()
    tdse_lib.set_device_memory_limit(used + 4 * 16 * B * (lmax + 1) * n + 65536)    # the batch's own vectors, no digits
    try:
        c = torch.from_numpy(C.copy()).cuda()
        H.propagate_batch(c, torch.from_numpy(F).cuda(), B, dt, steps)
        H.sync()
    finally:
        tdse_lib.set_device_memory_limit(0)
    H.close()
    for b in range(B):
        ref, _ = oracle.rk4(lmax, n, E, U, C[b], F[b], dt, steps)
        assert np.linalg.norm(c[b].cpu().numpy() - ref) < tol * np.linalg.norm(ref), b


def radial(n, lmax, R):
    """Hydrogen in a sphere of radius R on a sine grid: the dipole blocks of the lowest lmax + 1 angular momenta."""
    h = R / (n + 1)
    r = h * np.arange(1, n + 1)
    q = np.arange(1, n + 1)
    S = np.sqrt(2.0 / (n + 1)) * np.sin(np.outer(q, q) * np.pi / (n + 1))
    T = S @ np.diag((q * np.pi / R) ** 2 / 2) @ S
    V = [np.linalg.eigh(T + np.diag(l * (l + 1) / (2 * r * r) - 1 / r))[1] for l in range(lmax + 1)]
    return np.stack([(V[l].T * r) @ V[l + 1] * ((l + 1) / np.sqrt((2 * l + 1) * (2 * l + 3))) for l in range(lmax)])


# Largest error of a component over the sum of its own terms' magnitudes that the products these replace showed
# on the same states: FP32 sums of n products, any order (n 2^-24 each part); float-float sums, twice the 4.3e-7
# measured (offset sums, exact to 2^-46 of the largest product); FP64 sums (n 2^-53 each part).
def own_bound(prec, n):
    return {"fp32": (2 * n + 4) * 2.0 ** -24, "df32": 2.0 ** -20, "fp64": (2 * n + 2) * 2.0 ** -53}[prec]


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
@pytest.mark.parametrize("what", ["dominant", "hydrogen"])
def test_small_components_keep_their_digits(tdse_lib, prec, what):
    """Bound states: one amplitude near 1, the others of its block far below it."""
    lmax, n, B = 3, 301, 8
    rng = np.random.default_rng(9)
    x = np.zeros((lmax + 1, n), np.complex128)
    if what == "dominant":
        # dipole elements of the dominant amplitude that fall to 1e-7, a tail of 1e-10
        U = rng.standard_normal((lmax, n, n)) / np.sqrt(n)
        fall = (1.0 + np.arange(n) / 5.0) ** -4
        U[:, :, 0] *= fall
        U[:, 0, :] *= fall
        x[:] = 1e-10 * (rng.standard_normal(x.shape) + 1j * rng.standard_normal(x.shape))
        x[:, 0] = 1.0
    else:
        # the ground state and the first orders of perturbation theory in a weak field
        U = radial(n, lmax, 100.0)
        x[0, 0] = 1.0
        term = x.copy()
        for order in range(1, 6):
            y = np.zeros_like(x)
            y[:-1] += np.einsum("lij,lj->li", U, term[1:])
            y[1:] += np.einsum("lij,li->lj", U, term[:-1])
            term = -1j * 10.0 ** -order * y
            x += term
    U = U.astype(np.float32).astype(np.float64) if prec == "fp32" else U
    ref, own = np.zeros(x.shape, np.clongdouble), np.zeros(x.shape)
    for l in range(lmax):
        u = U[l].astype(np.longdouble)
        ref[l] += u @ x[l + 1].real + 1j * (u @ x[l + 1].imag)
        ref[l + 1] += u.T @ x[l].real + 1j * (u.T @ x[l].imag)
        own[l] += (np.abs(u) @ np.abs(x[l + 1])).astype(float)
        own[l + 1] += (np.abs(u).T @ np.abs(x[l])).astype(float)
    # one Taylor term in a field of 2^60, beside which the states themselves vanish
    F = 2.0 ** 60
    H = tdse_lib.Hamiltonian(np.zeros(x.size), U, lmax, n, prec)
    c = torch.from_numpy(np.stack([x.reshape(-1)] * B)).cuda()
    H.propagate_batch(c, torch.full((B, 2), F, dtype=torch.float64, device="cuda"), B, 1.0, 1, "taylor", order=1)
    H.sync()
    H.close()
    for b in range(B):
        got = (c[b].cpu().numpy().reshape(x.shape).astype(np.clongdouble) - x) * 1j / np.longdouble(F)
        err = np.abs(got - ref).astype(np.float64)
        assert np.all(err <= own_bound(prec, n) * own), float((err / own).max())


def run_batch(H, B, steps, dt=0.01):
    N = H.N
    c = torch.from_numpy(np.stack([inputs.random_state(N, b) for b in range(B)])).cuda()
    H.propagate_batch(c, torch.full((B, steps + 1), 0.1, dtype=torch.float64, device="cuda"), B, dt, steps)
    H.sync()


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
def test_the_workspace_does_not_grow_with_the_steps(tdse_lib, prec):
    lmax, n, B = 2, 100, 16
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, prec)
    run_batch(H, B, 2)
    used = tdse_lib.device_memory_in_use()
    run_batch(H, B, 200)
    assert tdse_lib.device_memory_in_use() == used
    H.close()


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
def test_no_workspace_of_digits_stays_where_the_other_path_serves(tdse_lib, prec):
    """Under a cap that leaves the digits no room, a batch holds what the pipe kernels need and no more, so
    that a cap of just that serves it (what the digits took first would be missing)."""
    lmax, n, B = 2, 200, 64
    N = (lmax + 1) * n
    words = {"fp32": 2, "df32": 4, "fp64": 0}[prec]               # of four bytes, twice: the products' inputs
    own = 2 * 16 * B * N + 2 * 4 * words * B * N + 3 * 2 * 4 * B if prec != "fp64" else 4096
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, prec)
    used = tdse_lib.device_memory_in_use()
    tdse_lib.set_device_memory_limit(used + own)
    try:
        run_batch(H, B, 2)
        assert tdse_lib.device_memory_in_use() <= used + own
    finally:
        tdse_lib.set_device_memory_limit(0)
    H.close()


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
def test_other_calls_get_the_digits_memory(tdse_lib, prec):
    """A call that runs out of memory while its context holds digits succeeds without them."""
    lmax, n, B, steps = 2, 200, 64, 8
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, prec)
    before = tdse_lib.device_memory_in_use()
    c0 = torch.from_numpy(inputs.random_state(H.N, 1)).cuda()
    F = torch.full((steps + 1,), 0.1, dtype=torch.float64, device="cuda")
    w = torch.ones(H.N, dtype=torch.float64, device="cuda")
    want = H.adjoint(c0, F, 0.01, steps, w)[0].clone()
    need = tdse_lib.device_memory_in_use() - before
    H.close()
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, prec)
    run_batch(H, B, 2)
    held = tdse_lib.device_memory_in_use()
    tdse_lib.set_device_memory_limit(held + need // 2)
    try:
        got = H.adjoint(c0, F, 0.01, steps, w)[0]
        assert torch.equal(got, want)
        assert tdse_lib.device_memory_in_use() < held
    finally:
        tdse_lib.set_device_memory_limit(0)
    H.close()


@pytest.mark.parametrize("prec", ["fp32", "df32", "fp64"])
def test_a_captured_batch_outlives_later_calls(tdse_lib, prec):
    """A batch recorded in a caller's graph replays on the memory it was recorded with: after a larger batch
    of the same context, after one of another tile and after a call that ran out of memory."""
    lmax, n, B, steps, dt = 2, 200, 16, 2, 0.01
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, prec)
    c0 = torch.from_numpy(np.stack([inputs.random_state(H.N, b) for b in range(B)])).cuda()
    F = torch.full((B, steps + 1), 0.1, dtype=torch.float64, device="cuda")
    c = c0.clone()
    H.propagate_batch(c, F, B, dt, steps)
    H.sync()
    want = c.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        H.propagate_batch(c, F, B, dt, steps)

    def replay():
        c.copy_(c0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(c, want)

    replay()
    for other in (3, 200, 3):
        run_batch(H, other, 1)
        replay()
    used = tdse_lib.device_memory_in_use()
    tdse_lib.set_device_memory_limit(used + 1024)
    try:
        with pytest.raises(tdse_lib.TDSEError):
            H.adjoint(c0[0], F[0], dt, steps, torch.ones(H.N, dtype=torch.float64, device="cuda"))
        assert tdse_lib.device_memory_in_use() >= used
    finally:
        tdse_lib.set_device_memory_limit(0)
    replay()
    del g
    H.close()


@pytest.mark.parametrize("lmax,n,few,many", [(3, 50, 11, 12), (7, 100, 7, 8), (3, 301, 5, 6)])
def test_few_fp64_pulses_run_one_by_one(tdse_lib, lmax, n, few, many):
    """Below the number of pulses from which the digit products pay, a stage of an FP64 batch takes no launch
    of its own (the kernels of one system hold all stages); above, it takes two.  Both give the same states."""
    steps, dt = 20, 0.01
    E, U = inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8)
    H = tdse_lib.Hamiltonian(E, U, lmax, n, "fp64")
    C = np.stack([inputs.random_state(H.N, b) for b in range(many)])
    F = torch.full((many, steps + 1), 0.1, dtype=torch.float64, device="cuda")
    out = []
    for B in (few, many):
        H.profile_read()
        c = torch.from_numpy(C[:B].copy()).cuda()
        H.propagate_batch(c, F[:B].clone(), B, dt, steps)
        launches = H.profile_read()[2]
        assert launches <= 4 * B + 4 if B == few else launches >= 8 * steps
        out.append(c.cpu().numpy())
    # 80 stages, each rounding once: the states agree to their FP64 rounding
    assert np.linalg.norm(out[0] - out[1][:few]) <= 80 * 2.0 ** -52 * np.linalg.norm(out[0])
    H.close()


def test_observables_get_the_digits_memory(tdse_lib):
    lmax, n, B = 2, 200, 64
    H = tdse_lib.Hamiltonian(inputs.energies(lmax, n), inputs.dipoles(lmax, n, 8), lmax, n, "df32")
    run_batch(H, B, 1)
    c = torch.from_numpy(np.stack([inputs.random_state(H.N, b) for b in range(B)])).cuda()
    held = tdse_lib.device_memory_in_use()
    tdse_lib.set_device_memory_limit(held + 16)
    try:
        norms = H.norm(c, B).cpu().numpy()
    finally:
        tdse_lib.set_device_memory_limit(0)
    assert np.allclose(norms, 1.0, rtol=0, atol=1e-12) and tdse_lib.device_memory_in_use() < held
    H.close()
