"""Rows of 128 .. 2048 elements on the n = 4096 kernels (several rows as one of 4096): against the oracle at sizes where the
last joint row is whole, holds a single row and lacks a single row, with guard bytes around every output; the rules are
in parity.py.  The row counts are above the sizes from which every one of these kernels is taken."""
import math

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


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_rows_of_any_magnitude(n, dtype):
    """Rows up to 1e36 through angles with small cosines, where values divided by the cosines' product overflow on the way: right
    all the same, in whole and in short joint rows and several in one, and the rows beside them the same bits as without."""
    theta = synth.angles(n, "uniform", 3)
    theta[1:3, ::3] = math.pi / 2 - 1e-5
    theta[3, ::5] = math.pi / 2 - 1e-3
    rows = 4096 // n * 700 + 1
    x = synth.rows(rows, n, "normal", 4, dtype=dtype)
    large = {0: 1e20, 1: 1e34, 4: 1e30, 9: 1e36, rows // 2: 1e28, rows - 1: 1e35}
    big = x.clone()
    for r, m in large.items():
        big[r] = x[r] * m
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    assert p.stage_form() & 1 == 0  # the scaled form
    th64, b64 = to_f64(theta), to_f64(big)
    amax = np.abs(b64).max(axis=1)
    y_ref, x_ref = oracle.forward(th64, b64), oracle.inverse(th64, b64)
    keep = torch.tensor([r not in large for r in range(rows)], device=DEV)
    y, xr = Guarded((rows, n), dtype, DEV), Guarded((rows, n), dtype, DEV)
    check_rows_close(p.forward(big.to(DEV), out=y.view), y_ref, amax, "forward")
    check_rows_close(p.inverse(big.to(DEV), out=xr.view), x_ref, amax, "inverse")
    assert torch.equal(y.view[keep], p.forward(x.to(DEV))[keep]) and torch.equal(xr.view[keep], p.inverse(x.to(DEV))[keep])
    if dtype == torch.bfloat16:
        check_rows_close(p.inverse(big.to(DEV), out_dtype=torch.float32), x_ref, amax, "inverse, fp32 out")
    for bits in (2, 4, 8):
        codes, scales = Guarded((rows, n * bits // 8), torch.uint8, DEV), Guarded((rows,), torch.float16, DEV)
        p.forward_quant(big.to(DEV), bits, codes.view, scales.view)
        check_quant(codes.view[keep], scales.view[keep], y_ref[keep.cpu().numpy()], bits, f"{bits} bits")
        for r in large:  # saturated: the lowest or the highest code, wherever the value is more than rounding noise
            assert scales.view[r] == 65504
            c = oracle.unpack(codes.view[r:r + 1].cpu().numpy(), bits)[0]
            sure = np.abs(y_ref[r]) > 1e-5 * amax[r]
            assert np.array_equal(c[sure], np.where(y_ref[r] > 0, 2 ** (bits - 1) - 1, -(2 ** (bits - 1)))[sure])
        plain = p.forward_quant(x.to(DEV), bits)
        assert torch.equal(codes.view[keep], plain[0][keep]) and torch.equal(scales.view[keep], plain[1][keep])
        assert codes.intact() and scales.intact()
        kept = p.fold_weights(big.to(DEV), bits, want_rotated=True)
        assert torch.equal(kept[0], codes.view) and torch.equal(kept[1], scales.view) and torch.equal(kept[2], y.view)
    assert y.intact() and xr.intact() and p.device_status() == 0


@pytest.mark.parametrize("n", [128, 256, 2048])
def test_infinities_and_nan_as_in_the_kernels_for_every_n(n, monkeypatch):
    """What the rotation by cos and sin makes of them, with the saturated scale of an infinite row; the rows beside them are the
    same bits as without."""
    rows = 4096 // n * 5 + 1
    p = Plan(n, DEV)
    p.set_angles(synth.angles(n, "normal", 1).to(DEV))
    x = synth.rows(rows, n, "normal", 2)
    clean = x.clone()
    x[3, 5], x[7, 1], x[rows - 1, 100] = float("inf"), float("nan"), float("-inf")
    x[9] = float("inf")
    run = lambda v: (p.forward(v.to(DEV)), p.inverse(v.to(DEV)), *(t for b in (2, 4, 8) for t in p.forward_quant(v.to(DEV), b)))
    got = run(x)
    others = [r for r in range(rows) if r not in (3, 7, 9, rows - 1)]
    for a, b in zip(got, run(clean)):
        assert torch.equal(a[others], b[others])
    monkeypatch.setenv("BFQ_GENERIC_ONLY", "1")
    for a, b in zip(got, run(x)):
        for r in (3, 7, 9, rows - 1):
            assert torch.equal(a[r].nan_to_num(), b[r].nan_to_num())
    assert got[3][3] == 65504


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype,kept", [(torch.float32, torch.float32), (torch.bfloat16, torch.bfloat16), (torch.bfloat16, torch.float32)])
def test_a_fold_that_keeps_its_rows_gives_the_bits_of_the_calls_that_give_one_of_them(n, dtype, kept):
    p = Plan(n, DEV)
    theta = synth.angles(n, "uniform", 3)
    p.set_angles(theta.to(DEV))
    W = synth.rows((1 << 20) // n + 1, n, "normal", 4, scale=0.02, dtype=dtype)
    y_ref = oracle.forward(to_f64(theta), to_f64(W))
    for bits in (2, 4, 8):
        codes, scales, rows = p.fold_weights(W.to(DEV), bits, want_rotated=True, rotated_dtype=kept)
        alone = p.fold_weights(W.to(DEV), bits)
        assert torch.equal(codes, alone[0]) and torch.equal(scales, alone[1])
        assert torch.equal(rows, p.forward(W.to(DEV), out_dtype=kept))
        check_quant(codes, scales, y_ref, bits, f"{bits} bits")
        check_rows_close(rows, y_ref, np.abs(to_f64(W)).max(axis=1), "rows")


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_an_output_with_a_row_stride_has_the_bits_of_a_contiguous_one(n, dtype):
    rows = (1 << 22) // n + 1
    p = Plan(n, DEV)
    p.set_angles(synth.angles(n, "uniform", 3).to(DEV))
    x = synth.rows(rows, n, "normal", 4, dtype=dtype).to(DEV)
    x[2] *= 1e37  # done again
    x[rows - 1, 3] = float("inf")
    for call in (p.forward, p.inverse):
        ref = call(x)
        for pad in (8, 4096):
            wide = Guarded((rows, n + pad), dtype, DEV)
            untouched = wide.view[:, n:].clone()
            call(x, out=wide.view[:, :n])
            same = lambda a, b: torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
            assert same(wide.view[:, :n], ref) and same(wide.view[:, n:], untouched) and wide.intact()
    assert p.device_status() == 0


@pytest.mark.parametrize("n", [128, 2048, 4096])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_a_single_row_may_have_any_row_stride(n, dtype):
    p = Plan(n, DEV)
    p.set_angles(synth.angles(n, "normal", 3).to(DEV))
    x = synth.rows(1, n, "normal", 4, dtype=dtype).to(DEV)
    far = x.as_strided((1, n), (1 << 41, 1))
    assert torch.equal(p.forward(far), p.forward(x)) and torch.equal(p.inverse(far), p.inverse(x))
    out = torch.empty_like(x)
    p.forward(x, out=out.as_strided((1, n), (1 << 41, 1)))
    assert torch.equal(out, p.forward(x))
    assert all(torch.equal(a, b) for a, b in zip(p.forward_quant(far, 4), p.forward_quant(x, 4)))


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_angles_that_need_the_three_shear_form(n, dtype):
    """Three stages of cosines of 1e-7: the factors leave the scaled form's range, forward and inverse (its own table layout)."""
    theta = synth.angles(n, "normal", 6)
    theta[2:5] = math.pi / 2 - 1e-7
    rows = ((1 << 21) + (1 << 12) if n == 128 else 1 << 19) // n + 3
    x = synth.rows(rows, n, "student_t3", 5, outliers=4, outlier_scale=20.0, dtype=dtype)
    x[4] *= 1e-30  # scale 0
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    th64, x64 = to_f64(theta), to_f64(x)
    amax = np.abs(x64).max(axis=1)
    y_ref = oracle.forward(th64, x64)
    y, xr = Guarded((rows, n + 8), dtype, DEV), Guarded((rows, n), dtype, DEV)
    check_rows_close(p.forward(x.to(DEV), out=y.view[:, :n]), y_ref, amax, "forward")
    check_rows_close(p.inverse(x.to(DEV), out=xr.view), oracle.inverse(th64, x64), amax, "inverse")
    for bits in (2, 4, 8):
        codes, scales, kept = p.fold_weights(x.to(DEV), bits, want_rotated=True)
        check_quant(codes, scales, y_ref, bits, f"{bits} bits")
        assert torch.equal(kept, y.view[:, :n])
    assert y.intact() and xr.intact() and p.stage_form() == 3 and p.device_status() == 0


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("upper", [True, False])
def test_an_overflow_in_one_element_of_the_last_stage(n, dtype, upper):
    """Small factors in one half of the row only: of a pair of the forward's last stage one quotient overflows, the other
    does not."""
    theta = synth.angles(n, "zero", 1)
    half = slice(n // 4, None) if upper else slice(0, n // 4)
    theta[2:4, half] = math.pi / 2
    theta[-1] = 0.5
    x = synth.rows(4096 // n * 3, n, "normal", 4, dtype=dtype)
    x[1, (slice(0, n // 2) if upper else slice(n // 2, None))] *= 1e30
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    assert p.stage_form() & 1 == 0
    th64, x64 = to_f64(theta), to_f64(x)
    amax = np.abs(x64).max(axis=1)
    y_ref = oracle.forward(th64, x64)
    check_rows_close(p.forward(x.to(DEV)), y_ref, amax, "forward")
    check_rows_close(p.inverse(x.to(DEV)), oracle.inverse(th64, x64), amax, "inverse")
    assert torch.equal(p.forward_quant(x.to(DEV), 8)[1][1], torch.tensor(65504.0, dtype=torch.float16, device=DEV))


@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("dtype,bits", [(torch.float32, 8), (torch.bfloat16, 4), (torch.float32, 2)])
def test_statistics_count_the_codes_of_the_call_without_them(n, dtype, bits):
    rows = (1 << 20) // n + 3
    p = Plan(n, DEV)
    theta = synth.angles(n, "uniform", 3)
    p.set_angles(theta.to(DEV))
    x = synth.rows(rows, n, "student_t3", 4, dtype=dtype)
    x[5] = 0.0
    codes, scales, hist, moments = p.forward_quant_stats(x.to(DEV), bits)
    plain = p.forward_quant(x.to(DEV), bits)
    assert torch.equal(codes, plain[0]) and torch.equal(scales, plain[1])
    assert np.array_equal(hist.cpu().numpy(), oracle.code_histogram(oracle.unpack(codes.cpu().numpy(), bits), bits))
    np.testing.assert_allclose(to_f64(moments), oracle.row_moments(oracle.forward(to_f64(theta), to_f64(x))), rtol=2e-5)


@pytest.mark.parametrize("n,rows", [(128, 4096), (1024, 700), (4096, 300)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_backward_where_the_scaled_sums_overflow(n, rows, dtype):
    """Rows of x near the end of fp32's range: stored over a product of cosines they overflow, the sums of d-theta do not.  The
    CTAs that meet them take their rows again; dx of the other rows is the same bits."""
    p, theta, x, xd = inputs(n, rows, dtype)
    g = synth.rows(rows, n, "normal", 5, dtype=dtype)
    plain = p.backward(xd, g.to(DEV))[0]
    for r in (3, rows // 2):
        x[r] *= 2.0 ** 110
        g[r] *= 2.0 ** -20
    xd.copy_(x)
    dx, dth = p.backward(xd, g.to(DEV))
    dx_ref, dth_ref = oracle.backward(to_f64(theta), to_f64(x), to_f64(g))
    check_rows_close(dx, dx_ref, np.abs(to_f64(g)).max(axis=1), "dx")
    check_dtheta(dth, dth_ref, "dtheta")
    keep = torch.ones(rows, dtype=torch.bool, device=DEV)
    keep[3] = keep[rows // 2] = False
    assert torch.equal(dx[keep], plain[keep]) and p.device_status() == 0


@pytest.mark.parametrize("n,rows,over", [(4096, 301, "g"), (4096, 301, "x"), (512, 3001, "x")])
def test_backward_into_its_own_input(n, rows, over):
    """dx over g or x (no CTA may need its rows a second time then): the results of separate buffers, to rounding."""
    p, theta, x, xd = inputs(n, rows, torch.float32)
    gd = synth.rows(rows, n, "normal", 5).to(DEV)
    dx, dth = p.backward(xd, gd)
    dx2, dth2 = p.backward(xd, gd, dx=gd if over == "g" else xd)
    assert (dx2 - dx).abs().max() <= 1e-5 * dx.abs().max() and (dth2 - dth).norm() <= 1e-5 * dth.norm()
    assert p.device_status() == 0


@pytest.mark.parametrize("n,rows", [(4096, 1001), (256, 20001), (128, 40000)])
@pytest.mark.parametrize("over", ["g", "x"])
def test_backward_into_its_own_bf16_input(n, rows, over):
    """The same where the group of threads that brings g down writes dx, before another has read the row of x that may lie there:
    several rows for each CTA.  (Both are fp32 results rounded to bf16: an ulp, 2^-7, apart at most.)"""
    p, theta, x, xd = inputs(n, rows, torch.bfloat16)
    gd = synth.rows(rows, n, "normal", 5, dtype=torch.bfloat16).to(DEV)
    dx, dth = p.backward(xd, gd)
    dx2, dth2 = p.backward(xd, gd, dx=gd if over == "g" else xd)
    a, b = dx.float(), dx2.float()
    assert ((a - b).abs() <= 2.0 ** -7 * a.abs() + 1e-5 * a.abs().max()).all() and (dth2 - dth).norm() <= 1e-5 * dth.norm()
    assert p.device_status() == 0


def test_backward_rounds_each_row_once_into_the_sums():
    """d-theta against 64 bits (n = 4096).  A running sum of m rows with one rounding each is off by 2.5e-8 sqrt(m / 2) of the total (the
    mean square of a rounding to 24 bits, the sum growing as a random walk), 4.3e-7 here with the 2e-7 that the rows' own rounding
    gives; with two roundings per row it is 5.7e-7."""
    n, rows = 4096, 65536
    theta = synth.angles(n, "normal", 1)
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    x = synth.rows(rows, n, "student_t3", 3, outliers=8, outlier_scale=50.0, dtype=torch.bfloat16, device=DEV)
    g = synth.rows(rows, n, "normal", 4, dtype=torch.bfloat16, device=DEV)
    dth = p.backward(x, g)[1].double()
    th = theta.to(DEV).double()
    ref = torch.zeros_like(dth)
    for r in range(0, rows, 16384):
        u, v = x[r:r + 16384].double(), g[r:r + 16384].double()

        def turn(w, s, back):
            lo, hi = w.view(-1, n >> (s + 1), 2, 1 << s).unbind(2)
            c, sn = torch.cos(th[s]).view(-1, 1 << s), torch.sin(th[s]).view(-1, 1 << s) * (-1 if back else 1)
            return torch.stack((c * lo - sn * hi, sn * lo + c * hi), 2).view(-1, n)
        for s in range(12):
            u = turn(u, s, False)
        for s in reversed(range(12)):
            (ul, uh), (vl, vh) = (w.view(-1, n >> (s + 1), 2, 1 << s).unbind(2) for w in (u, v))
            ref[s] += (vh * ul - vl * uh).sum(0).reshape(-1)
            u, v = turn(u, s, True), turn(v, s, True)
    assert (dth - ref).norm() <= 4.9e-7 * ref.norm()
    assert p.device_status() == 0


@pytest.mark.parametrize("exponent", [-118, 0, 95])
@pytest.mark.parametrize("n,rows", [(4096, 300), (1024, 700), (128, 4096)])
def test_backward_at_either_end_of_the_range(n, rows, exponent):
    """g at 2^exponent with angles whose cosines multiply to 2^-38, close to the least factor of the scaled form: g goes through the
    stages times its factor, and must come out with all its bits where that product would be subnormal.  (At 2^95 it overflows on the
    way and the rows are done again.)"""
    log_n = n.bit_length() - 1
    sign = torch.randint(0, 2, (log_n, n // 2), generator=torch.Generator().manual_seed(1)) * 2 - 1
    theta = (sign * math.acos(2.0 ** (-38 / log_n))).float()
    p = Plan(n, DEV)
    p.set_angles(theta.to(DEV))
    x = synth.rows(rows, n, "normal", 2)
    g = synth.rows(rows, n, "normal", 3) * 2.0 ** exponent
    dx, dth = p.backward(x.to(DEV), g.to(DEV))
    dx_ref, dth_ref = oracle.backward(to_f64(theta), to_f64(x), to_f64(g))
    check_rows_close(dx, dx_ref, np.abs(to_f64(g)).max(axis=1), "dx")
    check_dtheta(dth, dth_ref, "dtheta")
    assert p.device_status() == 0


@pytest.mark.parametrize("n,rows", [(4096, 700), (1024, 3000), (128, 40000)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_backward_with_an_infinity_in_g(n, rows, dtype):
    """An infinity or NaN in a row of g leaves no angle's sum finite; beside it dx of a row that is only too large for the scaled form is
    right, and dx of every other row the same bits."""
    p, theta, x, xd = inputs(n, rows, dtype)
    g = synth.rows(rows, n, "normal", 5, dtype=dtype)
    plain = p.backward(xd, g.to(DEV))[0]
    other = torch.ones(rows, dtype=torch.bool, device=DEV)
    other[5] = other[rows - 2] = False
    for large in (False, True):
        g[5, 7], g[rows - 2, n - 1] = math.inf, math.nan
        if large:
            g[rows // 2] *= 2.0 ** 100
            other[rows // 2] = False
        dx, dth = p.backward(xd, g.to(DEV))
        assert torch.equal(dx[other], plain[other]) and not torch.isfinite(dth).any()
        assert not torch.isfinite(dx[5]).any() and torch.isnan(dx[rows - 2]).all()
        if large:
            row = g[rows // 2:rows // 2 + 1]
            check_rows_close(dx[rows // 2:rows // 2 + 1], oracle.inverse(to_f64(theta), to_f64(row)), np.abs(to_f64(row)).max(axis=1), "dx")
    assert p.device_status() == 0
