"""U Psi from 8-bit digits on the tensor cores (n >= 9) and in fixed point (n
<= 8) against complex128 numpy, at the sizes where a tile, a column block or a
split ends, on targets whose digits are all alike or mostly zero, and on inputs
outside the digits' scale (the FP64 kernel behind them).

Tolerance: numpy's own sum of 2^n products rounds by up to about 2^-53 sqrt(2
2^n) of the result; four times that, and 2^-50 for small n."""
import numpy as np
import pytest

from paper_2405_12866_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    with qfs.Context(0) as c:
        yield c


def _product(ctx, U, Psi, prec):
    import torch
    n = int(np.log2(U.shape[0]))
    out = ctx.target_product(n, torch.from_numpy(np.ascontiguousarray(U)).cuda(),
                             torch.from_numpy(np.ascontiguousarray(Psi)).cuda(), prec)
    return out.cpu().numpy()


def _check(got, U, Psi):
    ref = U @ Psi
    tol = max(2.0 ** -50, 4 * 2.0 ** -53 * np.sqrt(2 * U.shape[0]))
    for j in range(Psi.shape[1]):
        assert np.linalg.norm(got[:, j] - ref[:, j]) <= tol * max(np.linalg.norm(ref[:, j]), 1e-290), j


def _brick(n, layers=3):
    pairs = w.brick_pairs(n, layers)
    return w.target_unitary(w.haar_gates(5, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)


@pytest.mark.parametrize("n,M", [(2, 1), (2, 4), (3, 5), (5, 32), (6, 33), (6, 64), (7, 1), (7, 16), (7, 17), (7, 32),
                                 (7, 33), (8, 16), (9, 65), (10, 31)])
@pytest.mark.parametrize("prec", [0, 1])
def test_product_matches_numpy(ctx, n, M, prec):
    U, Psi = _brick(n), w.sample_states(6, n, M)
    _check(_product(ctx, U, Psi, prec), U, Psi)


@pytest.mark.parametrize("n", [5, 8])
@pytest.mark.parametrize("what", ["identity", "minus_identity", "hadamard", "hadamard_of_hadamard", "permutation", "basis_states"])
def test_product_of_structured_targets(ctx, n, what):
    N = 1 << n
    H = np.array([[1.0]])
    for _ in range(n):
        H = np.kron(H, np.array([[1, 1], [1, -1]]) / np.sqrt(2))
    Psi = w.sample_states(6, n, 8)
    U = {"identity": np.eye(N), "minus_identity": -np.eye(N), "hadamard": H, "hadamard_of_hadamard": H,
         "permutation": np.roll(np.eye(N), 3, axis=0), "basis_states": _brick(n)}[what].astype(np.complex128)
    if what == "hadamard_of_hadamard":
        Psi = H[:, :8].astype(np.complex128)
    if what == "basis_states":
        Psi = w.basis_states(3, n, 8)
    _check(_product(ctx, U, Psi, 0), U, Psi)


@pytest.mark.parametrize("n", [5, 8])
@pytest.mark.parametrize("what", ["target_times_2", "target_times_1e-9", "one_row_times_3", "columns_of_all_sizes", "no_states",
                                  "tiny_states", "huge_states"])
def test_product_of_inputs_without_unit_norms(ctx, n, what):
    U, Psi = _brick(n), w.sample_states(6, n, 8).copy()
    if what == "columns_of_all_sizes" and n >= 7:
        Psi *= np.array([1, 1e-200, 0, 1e100, 1e-3, 7, 1e8, 1])[None, :]
    elif what.endswith("_states"):
        Psi *= {"no": 0.0, "tiny": 1e-290, "huge": 1e290}[what.split("_")[0]]
    elif what == "one_row_times_3":
        U[3] *= 3
    elif what != "columns_of_all_sizes":
        U = U * float(what.rsplit("_", 1)[1])
    _check(_product(ctx, U, Psi, 0), U, Psi)


@pytest.mark.parametrize("n", [5, 8])
def test_product_passes_nan_and_inf_on(ctx, n):
    U, Psi = _brick(n), w.sample_states(6, n, 8)
    U[3, 5] = np.nan
    U[4, 1] = np.inf
    got = _product(ctx, U, Psi, 0)
    assert np.isnan(got[3]).all() and not np.isfinite(got[4]).any()
    assert np.isfinite(np.delete(got, [3, 4], axis=0)).all()


@pytest.mark.parametrize("n, M", [(2, 3), (3, 8), (5, 31), (6, 64), (7, 9), (7, 128), (8, 1), (8, 50)])
def test_small_product_column_by_column_and_row_by_row(ctx, n, M):
    """Up to 8 qubits: rows of U and columns of Psi of very different sizes in
    one block, each to FP64 accuracy of its own.  The exact product comes from
    integers: entries are multiples of 2^-20, scaled by powers of two.  A result
    rounds by 2^-53 twice at most, its inputs by 2^-56 of the row's and the
    column's largest entry times the sum of the others (2 2^n terms)."""
    N = 1 << n
    rng = np.random.default_rng(9)
    u, p = (rng.integers(-(1 << 20), 1 << 20, s).astype(np.int64) for s in ((2, N, N), (2, N, M)))
    ru, cp = rng.integers(-300, 300, (N, 1)), rng.integers(-200, 200, (1, M))
    U, Psi = np.ldexp(u * 2.0**-20, ru), np.ldexp(p * 2.0**-20, cp)
    want = np.ldexp((u[0] @ p[0] - u[1] @ p[1]) * 2.0**-40, ru + cp), np.ldexp((u[0] @ p[1] + u[1] @ p[0]) * 2.0**-40, ru + cp)
    got = _product(ctx, U[0] + 1j * U[1], Psi[0] + 1j * Psi[1], 0)
    size = np.abs(U).max(axis=(0, 2))[:, None] * np.abs(Psi).max(axis=(0, 1))[None, :]
    for g, e in zip((got.real, got.imag), want):
        assert np.all(np.abs(g - e) <= 2.0**-52 * np.abs(e) + 2 * N * 2.0**-55 * size)


@pytest.mark.parametrize("what", ["identity", "minus_identity", "hadamard", "hadamard_of_hadamard", "permutation", "basis_states"])
def test_digits_of_structured_targets(ctx, what):
    test_product_of_structured_targets(ctx, 9, what)


@pytest.mark.parametrize("what", ["target_times_2", "target_times_1e-9", "one_row_times_3", "columns_of_all_sizes", "no_states",
                                  "tiny_states", "huge_states"])
def test_digits_of_inputs_without_unit_norms(ctx, what):
    test_product_of_inputs_without_unit_norms(ctx, 9, what)


@pytest.mark.parametrize("M", [1, 16, 17, 32, 33])
def test_digits_match_numpy(ctx, M):
    test_product_matches_numpy(ctx, 9, M, 0)


def test_digits_pass_nan_and_inf_on(ctx):
    test_product_passes_nan_and_inf_on(ctx, 9)
