"""How far U Psi of the batched form is from the exact product, seen through
the costs it reports.

A problem's reported cost is |Phi - C Psi|^2 / M with Phi = U Psi + e as the
set-up computed it and C the circuit of the returned gates.  With r = U Psi - C
Psi in 80 bits, M (cost - |r|^2 / M) / (2 |r|) is the component of the error
along r, up to |e|^2 / |r|.  The targets are a brick wall plus noise of 1e-5, so
that r is a direction the gates do not reach, of about 2 N M real dimensions,
and the root mean square of that component over many problems is |e| / sqrt(2 N
M).

Bound: FP64 arithmetic forms a component of U Psi from 2 N products, each of
which rounds by 2^-54 of a partial sum on average, and C Psi carries the
rounding of the returned gates, about 2^-53 a gate; relative to |U Psi| that is
below 2^-51 each up to 6 qubits and 9 gates, 2^-50.5 together."""
import numpy as np
import pytest

from paper_2405_12866_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M", [(3, 4), (4, 8), (5, 16), (6, 16)])
def test_target_product_of_the_set_up_is_as_exact_as_fp64(n, M):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    P, N, pairs = 96, 1 << n, w.brick_pairs(n, 3)
    rng = np.random.default_rng(17)
    problems, samples, starts = [], [], []
    for i in range(P):
        g = w.haar_gates(100 + i, w.STREAM_TARGET_GATES, len(pairs))
        noise = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
        problems.append((n, pairs, w.target_unitary(g, pairs, n) + 1e-5 / np.sqrt(2 * N) * noise))
        samples.append(w.sample_states(200 + i, n, M))
        starts.append(g[None])
    prm = qfs.default_params(M=M, multistarts=1, max_sweeps=2, dist_tol=1e-30, refine_sweeps_max=0, precision=qfs.QFS_MIXED)
    with qfs.Context(0) as ctx:
        gates, info = ctx.instantiate_batch(problems, prm, samples, starts)
    along = []
    for (_, _, U), Psi, g, r in zip(problems, samples, gates, info):
        C = Psi.astype(np.clongdouble)
        for k, (a, b) in enumerate(pairs):
            T = np.moveaxis(C.reshape((2,) * n + (M,)), (a, b), (0, 1))
            T = np.einsum("xy,yz->xz", g[k].astype(np.clongdouble), T.reshape(4, -1)).reshape(T.shape)
            C = np.moveaxis(T, (0, 1), (a, b)).reshape(N, M)
        d = U.astype(np.clongdouble) @ Psi.astype(np.clongdouble) - C
        norm = np.sqrt(np.sum(d.real ** 2 + d.imag ** 2))
        assert 1e-6 < norm < 1e-3
        along.append(float((M * np.longdouble(r["cost"]) - norm ** 2) / (2 * norm)))
    rms = np.sqrt(np.mean(np.square(along)))
    assert rms <= 2.0 ** -50.5 * np.sqrt(M) / np.sqrt(2 * N * M), rms * np.sqrt(2 * N)
