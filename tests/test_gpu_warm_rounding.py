"""The roundings of the warm-start network's features and of its output gradient
next to the middle between two floats, where pairs of floats alone may round the
other way than FP64, and the loss against the exact sum."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 11


@pytest.fixture(scope="module")
def model():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    with qfs.Context(0) as c:
        m = qfs.WarmStart(c, seed=SEED, batch_cap=1152)
        yield m
        m.close()


def _beside_a_middle(b, rng, lo=-52, hi=-48):
    """a such that the exact a b is 2^lo .. 2^hi of it beside the middle between the
    float mid (itself the middle between two bf16, the lower one even) and the next:
    (a, mid or the float above it, whichever a b rounds to)."""
    while True:
        mid = np.float32(abs(b) * rng.uniform(0.6, 1.4))
        mid = np.uint32((mid.view(np.uint32) & 0xFFFE0000) | 0x8000).view(np.float32)
        up = np.uint32(mid.view(np.uint32) + 1).view(np.float32)
        tie = (Fraction(float(mid)) + Fraction(float(up))) / 2
        a = float(tie / Fraction(abs(b)))
        for a in a + np.spacing(a) * rng.permutation(np.arange(-8, 9)):
            off = Fraction(float(a)) * Fraction(abs(b)) / tie - 1
            if Fraction(2) ** lo <= abs(off) <= Fraction(2) ** hi:
                return math.copysign(float(a), b), (up if off > 0 else mid)


def test_features_beside_a_middle(model):
    """A target with one entry a row has features 4 a b, rounded to FP32 and to bf16.  The
    first layer's weight gradient of a single target is g_o X_k, exactly: its columns
    over a column of 1 give X."""
    from oracle import mlp_oracle as mo
    from paper_2405_12866_gb300 import qfs
    phi = qfs.generate_inputs(SEED ^ 0x5EEDF1C5, 4, 8, 1, 1)[0]  # (to the last bit)
    rng = np.random.default_rng(3)
    labels = rng.standard_normal((1, 192))
    for _ in range(40):
        U, want, cols = np.zeros((1, 16, 16), dtype=np.complex128), [], []
        U[0, 0, 0] = 0.25 / phi[0, 0].real  # feature 0 is 1
        for i in range(1, 16):
            q, j, im = rng.integers(16), rng.integers(8), rng.integers(2)
            b = phi[q, j].imag if im else phi[q, j].real
            U[0, i, q], r = _beside_a_middle(b, rng)
            want.append(float(mo.bf16(4 * r)))
            cols.append((i * 8 + j) * 2 + im)
        _, g = model.loss_grad(U, labels)
        gw = qfs.WarmStart.unflatten(g.astype(np.float64))[0][0]
        o = np.argmax(np.abs(gw[:, 0]))
        got = gw[o, cols] / gw[o, 0]
        assert np.all(np.abs(got - want) <= 1e-6 * np.abs(want)), (got, want)


def _bias_only(model, bias):
    """Parameters with which every output is its bias."""
    from paper_2405_12866_gb300 import qfs
    p = np.zeros_like(model.get_params())
    qfs.WarmStart.unflatten(p)[-1][1][:192] = bias
    model.set_params(p)


@pytest.mark.parametrize("count", [1, 64])
def test_output_gradient_beside_a_middle(model, count):
    """The bias gradient of the last layer, with one row different from its outputs, is that
    row's scale (Y - T) rounded to FP32 (Y - T exact in FP64)."""
    from paper_2405_12866_gb300 import qfs
    rng = np.random.default_rng(4)
    scale = 2.0 / (count * 192)
    kept = model.get_params()
    near = 0
    for _ in range(20):
        bias, T = np.zeros(192, dtype=np.float32), np.zeros(192, dtype=np.float32)
        for o in range(192):  # of many differences the one whose product lies next to a middle
            y = rng.uniform(0.5, 1.0, 4096).astype(np.float32)
            t = (rng.uniform(-1.0, 1.0, 4096) * 2.0 ** -rng.integers(1, 25, 4096)).astype(np.float32)
            v = scale * (y.astype(np.float64) - t.astype(np.float64))
            f = v.astype(np.float32)
            other = np.where(f < v, np.nextafter(f, np.float32(np.inf)), np.nextafter(f, np.float32(-np.inf)))
            away = np.abs(v - (f.astype(np.float64) + other.astype(np.float64)) / 2) / np.abs(v)
            k = np.argmin(np.where(away > 2.0**-52, away, 1.0))
            bias[o], T[o] = y[k], t[k]
            near += away[k] < 2.0**-34
        _bias_only(model, bias)
        labels = np.tile(bias.astype(np.float64), (count, 1))
        labels[count // 2] = T
        _, g = model.loss_grad(np.tile(np.eye(16, dtype=np.complex128), (count, 1, 1)), labels)
        want = (scale * (bias.astype(np.float64) - T.astype(np.float64))).astype(np.float32)
        assert np.array_equal(qfs.WarmStart.unflatten(g)[-1][1][:192], want)
    assert near > 1000
    model.set_params(kept)


@pytest.mark.parametrize("count", [1, 300, 1100])
def test_loss_is_that_of_fp64(model, count):
    """Differences and squares round by 2^-53 each and the sum, of 2e5 terms in
    threads, by little more: 2^-50 of the loss."""
    rng = np.random.default_rng(count)
    kept = model.get_params()
    bias, T = rng.standard_normal(192).astype(np.float32), rng.standard_normal((count, 192)).astype(np.float32)
    _bias_only(model, bias)
    loss, _ = model.loss_grad(np.tile(np.eye(16, dtype=np.complex128), (count, 1, 1)), T.astype(np.float64))
    d = bias.astype(np.longdouble) - T.astype(np.longdouble)
    want = np.sum(np.sort((d * d).ravel())) / (count * 192)
    assert abs(loss - want) <= 2.0**-50 * want
    model.set_params(kept)
