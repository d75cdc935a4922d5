"""Rows of 128 .. 2048 elements on the n = 4096 kernels (several rows as one of 4096): against the oracle at sizes where the
last joint row is whole, holds a single row and lacks a single row, with guard bytes around every output; the rules are
in parity.py.  The row counts are above the sizes from which every one of these kernels is taken."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_09679_b200 import Plan, synth
from parity import Guarded, check_dtheta, check_quant, check_rows_close, to_f64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def batch(n, tail, elems=1 << 20):
    joint = 4096 // n
    return elems // n + {"whole": 0, "one": 1, "lacks one": joint - 1}[tail]


def inputs(n, rows, dtype, kind="normal", pad=0):
    theta = synth.angles(n, kind, n + 1)
    x = synth.rows(rows, n, "student_t3", n + 2, outliers=4, outlier_scale=20.0, dtype=dtype)
    xd = torch.full((rows, n + pad), float("nan"), dtype=dtype, device=DEV)[:, :n] if pad else torch.empty((rows, n), dtype=dtype, device=DEV)
    xd.copy_(x)
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    return p, theta, x, xd


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("tail,kind,pad", [("whole", "normal", 0), ("one", "uniform", 16), ("lacks one", "hadamard", 0)])
def test_forward_and_inverse(n, dtype, tail, kind, pad):
    rows = batch(n, tail, (1 << 21) + (1 << 12) if n == 128 else 1 << 19)
    p, theta, x, xd = inputs(n, rows, dtype, kind, pad)
    th64, x64 = to_f64(theta), to_f64(x)
    amax = np.abs(x64).max(axis=1)
    y_ref = oracle.forward(th64, x64)
    for bits in (2, 4, 8):
        codes, scales = Guarded((rows, n * bits // 8), torch.uint8, DEV), Guarded((rows,), torch.float16, DEV)
        p.forward_quant(xd, bits, codes.view, scales.view)
        check_quant(codes.view, scales.view, y_ref, bits, f"{bits} bits")
        assert codes.intact() and scales.intact()
    y, xr = Guarded((rows, n), dtype, DEV), Guarded((rows, n), dtype, DEV)
    check_rows_close(p.forward(xd, out=y.view), y_ref, amax, "forward")
    check_rows_close(p.inverse(xd, out=xr.view), oracle.inverse(th64, x64), amax, "inverse")
    assert y.intact() and xr.intact()
    if dtype == torch.bfloat16:
        check_rows_close(p.inverse(xd, out_dtype=torch.float32), oracle.inverse(th64, x64), amax, "inverse, fp32 out")
    assert p.device_status() == 0


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("tail,kind", [("one", "normal"), ("lacks one", "uniform")])
def test_backward(n, dtype, tail, kind):
    rows = batch(n, tail, 1 << 23 if dtype == torch.bfloat16 and n <= 1024 else 1 << 20)
    p, theta, x, xd = inputs(n, rows, dtype, kind)
    g = synth.rows(rows, n, "normal", 5, dtype=dtype)
    dx = Guarded((rows, n), dtype, DEV)
    _, dth = p.backward(xd, g.to(DEV), dx=dx.view)
    dx_ref, dth_ref = oracle.backward(to_f64(theta), to_f64(x), to_f64(g))
    check_rows_close(dx.view, dx_ref, np.abs(to_f64(g)).max(axis=1), "dx")
    check_dtheta(dth, dth_ref, "dtheta")
    assert dx.intact() and torch.equal(dth, p.backward(xd, g.to(DEV), want_dx=False)[1])
    assert p.device_status() == 0


@pytest.mark.parametrize("n", [128, 2048])
@pytest.mark.parametrize("rows", [1, 3])
def test_a_few_rows(n, rows):
    """One short joint row: most of what is loaded lies past the batch."""
    p, theta, x, xd = inputs(n, rows, torch.bfloat16)
    y_ref = oracle.forward(to_f64(theta), to_f64(x))
    for bits in (2, 4, 8):
        codes, scales = Guarded((rows, n * bits // 8), torch.uint8, DEV), Guarded((rows,), torch.float16, DEV)
        p.forward_quant(xd, bits, codes.view, scales.view)
        check_quant(codes.view, scales.view, y_ref, bits)
        assert codes.intact() and scales.intact()


@pytest.mark.parametrize("n", [128, 2048])
def test_rows_do_not_touch_each_other(n):
    """A row of infinities and a row of NaN among ordinary ones: the others' results are the same bits."""
    rows = batch(n, "whole", 1 << 23)
    p, _, x, xd = inputs(n, rows, torch.bfloat16)
    spoilt = xd.clone()
    spoilt[5], spoilt[rows - 2] = float("inf"), float("nan")
    keep = torch.ones(rows, dtype=torch.bool, device=DEV)
    keep[5] = keep[rows - 2] = False
    for a, b in ((p.forward(xd), p.forward(spoilt)), (p.inverse(xd), p.inverse(spoilt)), (p.backward(xd, xd)[0], p.backward(spoilt, spoilt)[0]),
                 *zip(p.forward_quant(xd, 4), p.forward_quant(spoilt, 4))):
        assert torch.equal(a[keep], b[keep])


def near_ties(rows, n, bits, seed):
    """fp32 rows whose elements lie a few units in the last place from (k + 1/2) s, s the row's scale: where rounding once and
    rounding twice differ."""
    g = np.random.default_rng(seed)
    s = g.uniform(0.01, 1.0, (rows, 1)).astype(np.float16).astype(np.float32)
    qmax = 2 ** (bits - 1) - 1
    x = ((g.integers(-qmax, qmax, (rows, n)) + np.float32(0.5)) * s).astype(np.float32)
    for _ in range(3):
        x = np.where(g.random(x.shape) < 0.5, np.nextafter(x, np.float32(np.inf)), np.nextafter(x, np.float32(-np.inf)))
    x[:, :1] = qmax * s
    return torch.from_numpy(x)


@pytest.mark.parametrize("n", [128, 512, 2048])
@pytest.mark.parametrize("bits", [2, 4, 8])
def test_codes_of_a_row_do_not_depend_on_the_rows_beside_it(n, bits):
    """A row of zeros in every joint row, a saturated one in some, or a batch whose last joint row lacks a row: the other
    rows' codes are the same bits."""
    joint, rows = 4096 // n, (1 << 21) // n
    p = Plan(n, DEV)
    p.set_angles(synth.angles(n, "zero", 1).to(DEV))
    x = near_ties(rows, n, bits, 7).to(DEV)
    codes, scales = p.forward_quant(x, bits)
    other = x.clone()
    other[1::joint] = 0.0
    other[1::3 * joint] = 1e9
    keep = torch.ones(rows, dtype=torch.bool, device=DEV)
    keep[1::joint] = False
    codes2, scales2 = p.forward_quant(other, bits)
    assert torch.equal(scales[keep], scales2[keep]) and torch.equal(codes[keep], codes2[keep])
    codes3, scales3 = p.forward_quant(x[:rows - 1], bits)
    assert torch.equal(scales[:-1], scales3) and torch.equal(codes[:-1], codes3)
