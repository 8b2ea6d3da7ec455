"""GPU checks of the warm-start network's loss and gradients where its kernels
change their path: row counts around their 64-row tiles and 128-row padding,
targets with exact zeros and with entries outside the pair arithmetic's range
(one such target takes FP64 products, its neighbours do not)."""
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
    c = qfs.Context(0)
    yield c
    c.close()


def _targets(count, seed):
    """Haar-like unitaries; every third a permutation (exact zeros), every fifth with 1e-17 in place of its zeros."""
    rng = np.random.default_rng(seed)
    U = np.linalg.qr(rng.standard_normal((count, 16, 16)) + 1j * rng.standard_normal((count, 16, 16)))[0]
    for i in range(0, count, 3):
        U[i] = np.eye(16)[rng.permutation(16)]
        if i % 5 == 0:
            U[i] = U[i] + (U[i] == 0) * (1e-17 - 1e-17j)
    return np.ascontiguousarray(U)


@pytest.mark.parametrize("count", [63, 65, 128, 300, 1100])
def test_loss_and_gradients(ctx, count):
    from oracle import mlp_oracle as mo
    from paper_2405_12866_gb300 import qfs
    from paper_2405_12866_gb300 import workloads as w
    seed = 11
    model = qfs.WarmStart(ctx, seed=seed, batch_cap=1152)
    U = _targets(count, count)
    labels = np.random.default_rng(count + 1).standard_normal((count, 192))
    model.loss_grad(U[::-1], labels[::-1])  # (nothing of an earlier call may remain)
    loss, g = model.loss_grad(U, labels)
    params = qfs.WarmStart.unflatten(model.get_params().astype(np.float64))
    F = 4.0 * np.einsum("tij,jk->tik", U, w.sample_states(seed ^ 0x5EEDF1C5, 4, 8))
    X = np.stack([F.real, F.imag], axis=-1).reshape(count, 256)
    want_loss, want, mags = mo.loss_and_grads(params, X, labels, 192, round_bf16=True, magnitudes=True)
    assert abs(loss - want_loss) < 1e-3 * want_loss
    got = qfs.WarmStart.unflatten(g.astype(np.float64))
    # A term whose FP32 value lies next to a bf16 rounding boundary can round
    # the other way: one bf16 step, 2^-7, of each term's size at most.  (Sums
    # of many terms: a single row's entry has one factor that is itself a sum
    # with cancellation.)
    for li, ((gw, gb), (ww, wb), (mw, mb)) in enumerate(zip(got, want, mags)):
        for a, b, m in ((gw, ww, mw), (gb, wb, mb)):
            assert np.all(np.abs(a - b) <= 2.0 ** -7 * m + 1e-6 * np.max(m)), li
    model.close()


@pytest.mark.parametrize("size", [1e-30, 1e25])
def test_loss_of_differences_outside_the_pairs_range(ctx, size):
    """Labels far above, and differences far below, the outputs' size: the loss
    in FP64 of the FP32 labels."""
    from paper_2405_12866_gb300 import qfs
    model = qfs.WarmStart(ctx, seed=2, batch_cap=128)
    U = _targets(70, 3)
    params = model.get_params() * np.float32(0.0)
    model.set_params(params)
    labels = np.random.default_rng(4).standard_normal((70, 192)) * size
    loss, g = model.loss_grad(U, labels)
    t = labels.astype(np.float32).astype(np.float64)
    want = np.mean(t * t)  # (a network of zeros: Y = 0)
    assert abs(loss - want) <= 1e-12 * want
    bias = qfs.WarmStart.unflatten(g.astype(np.float64))[3][1][:192]
    terms = -2.0 * t / t.size
    # 70 FP32 terms added in FP32, each and every sum rounded to 2^-24.
    assert np.all(np.abs(bias - terms.sum(0)) <= 80 * 2.0 ** -24 * np.abs(terms).sum(0) + 1e-44)
    model.close()
