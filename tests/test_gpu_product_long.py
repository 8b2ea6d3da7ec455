"""U Psi from 8-bit digits (n >= 9, and n = 8 from 97 columns on) against exact integers, at the sizes where a
CTA runs through many chunks, a part of a chunk or a second column block, for
targets and states whose digits are all alike, so that the digits' sums grow as
fast as they can.

Entries are integers: of U times 2^-(22 + n/2) (rows of norm 1 to a few percent),
of Psi below 2^23 times 2^-23, so every digit is exact and no product of digits
is left out.  What rounds is the result (2^-53 of it) and its unit (2^-54 of the
column's scale, a split at a time; at most 32 splits).  Where all digits are
alike, sums of digits may pass 2^24 between two readings: 2^-52 at three of 256
products (d = 5) and 2^-48 per 4096 (d = 6).  Entries constant over a row and a
column have 53 bits: then the inputs round too, by 2^-55 of 1 a product each."""
import numpy as np
import pytest

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


SIZES = [(8, 97), (8, 256), (9, 5), (10, 16), (11, 1), (11, 17), (11, 65), (12, 32), (12, 33), (12, 300), (13, 20), (13, 64)]


# (12, 2048: more columns than the scratch holds at a time.)
@pytest.mark.parametrize("n,M,alike,rows", [(n, M, a, 0) for n, M in SIZES for a in (False, True)] + [(12, 2048, False, 0)]
                         + [(n, M, False, 40) for n, M in [(9, 5), (10, 31), (11, 65), (12, 300), (12, 2048)]])
def test_digits_against_exact_integers(ctx, n, M, alike, rows):
    """rows: each row of U times a power of two up to 2^+-rows (the second pass)."""
    import torch
    N = 1 << n
    gen = torch.Generator(device="cuda").manual_seed(100 * n + M)

    def ints(lo, hi, shape):
        return torch.randint(lo, hi, shape, generator=gen, device="cuda", dtype=torch.int64)

    one = int((0.5 if n % 2 else np.sqrt(0.5)) * (1 << 22))
    if alike:  # one value and sign for a row and for a column, but for the low bits
        u = torch.stack([one - ints(0, 1 << 16, (N, 1)) + ints(0, 1 << 10, (N, N)) for _ in range(2)])
        p = torch.stack([ints(1 << 22, (1 << 23) - 1024, (1, M)) + ints(0, 1 << 10, (N, M)) for _ in range(2)])
    else:
        a = int(one * np.sqrt(3.0))
        u, p = ints(-a, a + 1, (2, N, N)), ints(-(1 << 23) + 1, 1 << 23, (2, N, M))
    up = torch.randint(-rows, rows + 1, (N, 1), generator=gen, device="cuda")
    U = torch.complex(*(torch.ldexp(x.double(), up - (22 + n // 2)) for x in u))
    Psi = torch.complex(*(torch.ldexp(x.double(), torch.tensor(-23, device="cuda")) for x in p))
    got = ctx.target_product(n, U, Psi, 0).cpu().numpy()
    some = np.unique(np.concatenate([[0, 1, 127, 128, N - 128, N - 1], np.random.default_rng(n).integers(0, N, 18)]))
    u, p = u[:, torch.from_numpy(some).cuda()].cpu().numpy(), p.cpu().numpy()
    scale = np.ldexp(1.0, up.cpu().numpy()[some])
    unit = 2.0 ** -(45 + n // 2) * scale
    want = (u[0] @ p[0] - u[1] @ p[1]).astype(np.longdouble) * unit, (u[0] @ p[1] + u[1] @ p[0]).astype(np.longdouble) * unit
    slack = 2 * N * (3 / 256 * 2.0**-52 + 2.0**-48 / 4096) if alike else 0.0
    for g, e in zip((got[some].real, got[some].imag), want):
        assert np.all(np.abs(g - e) <= 2.0**-53 * np.abs(e) + (32 * 2.0**-55 + slack) * scale)


@pytest.mark.parametrize("prec", [0, 1])
def test_sweep_of_a_target_with_rows_of_all_sizes(ctx, prec):
    """A run's set-up takes the second pass too: one sweep at 9 qubits against the oracle, to
    the tolerances of FP64 and complex64 sweeps of states of norm 1, times U's norm."""
    from oracle import qfs_oracle as o
    from paper_2405_12866_gb300 import workloads as w
    n, M = 9, 8
    pairs = w.brick_pairs(n, 2)
    U = w.target_unitary(w.haar_gates(701, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    U *= np.random.default_rng(1).uniform(0.2, 3.0, (1 << n, 1))
    Psi, G = w.sample_states(702, n, M), w.initial_gates(703, 2, len(pairs))
    _, env, _ = ctx.sweep_once(n, pairs, U, Psi, G, prec)
    for s in range(2):
        r = o.sweep(U @ Psi, Psi, G[s], pairs, n)
        assert np.max(np.abs(env[s] - r.envs)) < 3.0 * (1e-4 if prec else 1e-10)


@pytest.mark.parametrize("n,M", SIZES)
def test_digits_of_constant_rows_and_columns(ctx, n, M):
    import torch
    N = 1 << n
    rng = np.random.default_rng(100 * n + M)
    c = (rng.uniform(0.93, 1.07, N) * np.exp(2j * np.pi * rng.uniform(size=N))) / np.sqrt(N)
    d = rng.uniform(0.5, 0.999, M) + 1j * rng.uniform(-0.999, 0.999, M)
    U = torch.from_numpy(c).cuda()[:, None].expand(N, N).contiguous()
    Psi = torch.from_numpy(d).cuda()[None, :].expand(N, M).contiguous()
    got = ctx.target_product(n, U, Psi, 1).cpu().numpy()
    cr, ci, dr, di = (x.astype(np.longdouble) for x in (c.real, c.imag, d.real, d.imag))
    want = N * (np.outer(cr, dr) - np.outer(ci, di)), N * (np.outer(cr, di) + np.outer(ci, dr))
    # (U's and Psi's entries are below 1; a quarter more for what is above.)
    tol = 2 * N * 2.0**-55 * (1.25 + np.abs(c).max())
    for g, e in zip((got.real, got.imag), want):
        assert np.all(np.abs(g - e) <= 2.0**-53 * np.abs(e) + tol)
