"""bfq_dequant_gemm (the dense products of the reconstruction loss, paper Sec. 3.4) against float64 numpy, operand kind
by operand kind.  Tolerances from the arithmetic: integer codes and bf16 numbers are exact operands; an fp32 number is
split into two bf16 terms, relative error <= 2^-17 per element; accumulation is fp32 over K terms.  So for every
output  |c - ref| <= (eA + eB + K 2^-24) sum_k |A(i, k)| |B(j, k)|  with e = 2^-17 for an fp32 operand and 0 otherwise
(+ one fp32 rounding of the result); the tests allow twice that."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_09679_b200 import GemmOperand, Plan, synth
from parity import to_f64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def make_codes(rows, k, bits, seed):
    """Codes + scales as bfq_forward_quant writes them, from the oracle's quantizer on random rows."""
    y = synth.rows(rows, k, "student_t3", seed, outliers=4, outlier_scale=20.0, dtype=torch.float32)
    codes, scales = oracle.quantize(to_f64(y), bits)
    packed = torch.from_numpy(oracle.pack(codes, bits))
    s16 = torch.from_numpy(scales.view(np.int16)).view(torch.float16)
    return packed, s16, oracle.dequantize(codes, scales)       # dequantized values, float64 [rows][k]


def operand(kind, rows, k, transposed, seed):
    """-> (GemmOperand on the device, float64 [rows][k] values, relative operand error)."""
    if kind in ("f32", "bf16"):
        dt = torch.float32 if kind == "f32" else torch.bfloat16
        v = synth.rows(rows, k, "normal", seed, dtype=dt)
        t = v.t().contiguous() if transposed else v
        return GemmOperand(t.to(DEV), transposed=transposed), to_f64(v), (2.0 ** -17 if kind == "f32" else 0.0)
    bits = int(kind[-1])
    if not transposed:
        packed, s16, val = make_codes(rows, k, bits, seed)
        return GemmOperand(packed.to(DEV), s16.to(DEV), bits), val, 0.0
    packed, s16, val = make_codes(k, rows, bits, seed)          # stored [K][rows]: scales per k
    return GemmOperand(packed.to(DEV), s16.to(DEV), bits, transposed=True), val.T.copy(), 0.0


def check(p, A, a64, ea, B, b64, eb, alpha=1.0):
    c = to_f64(p.dequant_gemm(A, B, alpha))
    ref = alpha * (a64 @ b64.T)
    k = a64.shape[1]
    bound = (ea + eb + (k + 2) * 2.0 ** -24) * abs(alpha) * (np.abs(a64) @ np.abs(b64).T)
    assert c.shape == ref.shape and np.isfinite(c).all()
    worst = (np.abs(c - ref) / np.maximum(2 * bound, 1e-300)).max()
    assert worst <= 1.0, worst
    assert p.device_status() == 0


KINDS = ["f32", "bf16", "codes2", "codes4", "codes8"]


@pytest.mark.parametrize("ka", KINDS)
@pytest.mark.parametrize("kb", KINDS)
@pytest.mark.parametrize("ta,tb", [(False, False), (False, True), (True, True)])
def test_every_operand_kind(ka, kb, ta, tb):
    m, n, k = 200, 136, 192            # ragged tiles in m and n, three K blocks
    # a transposed code operand packs its rows along the stored row: stored rows must stay 16-byte multiples
    if ta and ka.startswith("codes"):
        m = 256 if ka == "codes2" else 224
    if tb and kb.startswith("codes"):
        n = 192 if kb == "codes2" else 160
    p = Plan(256, DEV)
    A, a64, ea = operand(ka, m, k, ta, 900)
    B, b64, eb = operand(kb, n, k, tb, 901)
    check(p, A, a64, ea, B, b64, eb, alpha=0.5)


def test_exact_integer_product_of_two_code_operands():
    """W4A4: both operands codes along K -> an exact integer product times the two scales."""
    p = Plan(256, DEV)
    A, a64, _ = operand("codes4", 300, 4096, False, 910)
    B, b64, _ = operand("codes4", 260, 4096, False, 911)
    c = to_f64(p.dequant_gemm(A, B))
    ref = a64 @ b64.T
    assert np.abs(c - ref).max() <= 2.0 ** -22 * np.abs(ref).max()   # two roundings (scales) of an exact sum


@pytest.mark.parametrize("ka,kb,ta,tb", [("bf16", "codes2", False, False), ("codes4", "codes8", False, False),
                                         ("codes2", "codes4", False, False), ("bf16", "bf16", False, False),
                                         ("bf16", "codes4", True, True), ("f32", "codes8", False, True), ("f32", "codes2", True, True)])
@pytest.mark.parametrize("m,n,k", [(1, 256, 64),         # one row, one K block
                                   (32, 257, 1088),      # a tile's K shared by several pairs of CTAs, an odd number of blocks
                                   (130, 640, 448),      # half a K block left over on the integer path
                                   (1025, 5120, 192),    # more tiles than pairs, a ragged last one
                                   (290, 36864, 64)])    # several turns of a short ring per pair
def test_tile_edges(ka, kb, ta, tb, m, n, k):
    if ta:
        m = (m + 15) // 16 * 16                           # stored rows are 16-byte multiples
    if tb:
        n = (n + 63) // 64 * 64
    p = Plan(256, DEV)
    A, a64, ea = operand(ka, m, k, ta, 920)
    B, b64, eb = operand(kb, n, k, tb, 921)
    # scales folded into an fp32 operand: one more rounding to fp32
    check(p, A, a64, ea, B, b64, eb + (2.0 ** -24 if tb and ka == "f32" else 0.0))


@pytest.mark.parametrize("ka,kb,ta,tb", [("f32", "codes4", False, True), ("f32", "codes2", True, True), ("f32", "f32", False, False),
                                         ("bf16", "f32", True, True), ("f32", "bf16", True, False)])
def test_operands_split_beforehand(ka, kb, ta, tb):
    """The workspace form (a row length that is no multiple of 8, scales along and across the stored rows) gives the bits of
    the form without; a workspace that is too small is refused."""
    from paper_2509_09679_b200.binding import lib, _stream
    m, n, k = ((212 if ka == "f32" else 208) if ta else 201), (192 if tb and kb.startswith("codes") else 136), 4160
    p = Plan(256, DEV)
    A, a64, ea = operand(ka, m, k, ta, 940)
    B, b64, eb = operand(kb, n, k, tb, 941)
    check(p, A, a64, ea + 2.0 ** -24, B, b64, eb)
    size = lib().bfq_dequant_gemm_workspace(p._h, m, n, k, A.kind, int(ta), B.kind, int(tb))
    assert size > 0
    ptr = lambda t: t.data_ptr() if t is not None else None
    out = [torch.full((m, n), float("nan"), device=DEV) for _ in range(2)]
    room = torch.empty(size, dtype=torch.uint8, device=DEV)
    for c, ws, bytes_, status in ((out[0], None, 0, 0), (out[1], room.data_ptr(), size, 0), (out[1], room.data_ptr(), size - 1, -7)):
        assert status == lib().bfq_dequant_gemm_split(p._h, m, n, k, 1.0, ptr(A.data), A.kind, int(ta), A.ld, ptr(A.scales), ptr(B.data), B.kind, int(tb),
                                                      B.ld, ptr(B.scales), ptr(c), n, ws, bytes_, _stream(c))
    assert torch.equal(out[0], out[1]) and p.device_status() == 0


def test_fp32_operands_where_there_is_no_room_to_split_them(monkeypatch):
    p = Plan(256, DEV)
    A, a64, ea = operand("f32", 200, 4160, False, 950)
    B, b64, eb = operand("f32", 136, 4160, False, 951)
    split = p.dequant_gemm(A, B)
    real, refused = torch.empty, []

    def empty(*size, dtype=None, **kwargs):
        if dtype == torch.uint8:
            refused.append(size)
            raise torch.OutOfMemoryError("no room")
        return real(*size, dtype=dtype, **kwargs)

    monkeypatch.setattr(torch, "empty", empty)
    assert torch.equal(p.dequant_gemm(A, B), split) and len(refused) == 1
    check(p, A, a64, ea, B, b64, eb)


@pytest.mark.parametrize("ka", ["bf16", "codes2", "codes4", "codes8"])
@pytest.mark.parametrize("kb", ["codes2", "codes4", "codes8"])
@pytest.mark.parametrize("m,n,k", [(1, 16, 64), (8, 15, 192), (3, 4100, 1088), (9, 100, 4096), (64, 33, 64)])
def test_a_few_rows_against_codes(ka, kb, m, n, k):
    """One pass over the codes: one lane's part of K up to several turns of the warps, one to eight tiles of eight rows."""
    p = Plan(256, DEV)
    A, a64, ea = operand(ka, m, k, False, 930)
    B, b64, eb = operand(kb, n, k, False, 931)
    check(p, A, a64, ea, B, b64, eb, alpha=-1.5)


@pytest.mark.parametrize("abits,bbits", [(8, 8), (8, 2), (4, 4), (2, 8), (4, 8), (2, 2)])
def test_a_row_of_codes_times_codes_is_the_same_in_any_batch(abits, bbits):
    """An exact integer product: the same bits whether a few rows or many are multiplied, also where the sums pass 2^24."""
    k, n, m = 16384, 130, 200
    g = torch.Generator().manual_seed(5)
    a, b = (torch.randint(0, 256, (r, k * bits // 8), dtype=torch.uint8, generator=g).to(DEV) for r, bits in ((m, abits), (n, bbits)))
    if abits == bbits == 8:  # codes of 64 .. 127
        a, b = (a & 0x3F) | 0x40, (b & 0x3F) | 0x40
    sa, sb = (torch.rand(r, generator=g).half().to(DEV) for r in (m, n))
    p = Plan(256, DEV)
    B = GemmOperand(b, sb, bbits)
    whole = p.dequant_gemm(GemmOperand(a, sa, abits), B)
    from paper_2509_09679_b200.calibrate import unpack_codes
    exact = (unpack_codes(a, abits).double() @ unpack_codes(b, bbits).double().t()) * sa.double().unsqueeze(1) * sb.double()
    assert ((whole.double() - exact).abs() <= 2.0 ** -22 * exact.abs()).all()  # three roundings of an exact sum
    for few in (1, 8, 30):
        assert torch.equal(whole[:few], p.dequant_gemm(GemmOperand(a[:few], sa[:few].contiguous(), abits), B)), few


@pytest.mark.parametrize("k", [2 ** 17 - 64, 2 ** 17])
@pytest.mark.parametrize("m", [3, 70])
@pytest.mark.parametrize("bits,low", [(8, 0x80), (4, 0x88), (2, 0xAA)])
def test_lowest_codes_up_to_where_integers_end(k, m, bits, low):
    """The largest sums the integer path takes, and the first K that it does not take (there the sums are multiples of
    4^(bits - 1), exact in fp32 up to 2^24 of them)."""
    a, b = (torch.full((r, k * bits // 8), low, dtype=torch.uint8, device=DEV) for r in (m, 33))
    one = lambda r: torch.ones(r, dtype=torch.float16, device=DEV)
    p = Plan(256, DEV)
    c = p.dequant_gemm(GemmOperand(a, one(m), bits), GemmOperand(b, one(33), bits))
    assert (c == float(k) * 4.0 ** (bits - 1)).all() and p.device_status() == 0


@pytest.mark.parametrize("n", [1024, 1040])
def test_either_side_of_the_rule_for_a_few_rows(n):
    """64 rows are eight passes up to 8 n K = 2^25 and tiles above."""
    p = Plan(256, DEV)
    A, a64, ea = operand("bf16", 64, 4096, False, 960)
    B, b64, eb = operand("codes4", n, 4096, False, 961)
    check(p, A, a64, ea, B, b64, eb)


@pytest.mark.parametrize("m,n", [(200, 136), (4096, 2048)])
def test_either_side_of_the_rule_for_splitting_beforehand(m, n):
    """The last K at which an fp32 operand is split in the tiles and the first at which it is split by a pass of its own."""
    from paper_2509_09679_b200.binding import lib
    p = Plan(256, DEV)
    first = next(k for k in range(128, 1 << 14, 64) if lib().bfq_dequant_gemm_workspace(p._h, m, n, k, 0, 0, 1, 0) > 0)
    for k in (first - 64, first):
        A, a64, ea = operand("f32", m, k, False, 970)
        B, b64, eb = operand("bf16", n, k, False, 971)
        check(p, A, a64, ea, B, b64, eb)


def test_argument_validation():
    from paper_2509_09679_b200 import BfqError
    p = Plan(256, DEV)
    a = GemmOperand(torch.zeros((8, 100), device=DEV))
    b = GemmOperand(torch.zeros((8, 100), device=DEV))
    with pytest.raises(BfqError) as e:
        p.dequant_gemm(a, b)                                      # K not a multiple of 64
    assert e.value.status == -5
    c = p.dequant_gemm(GemmOperand(torch.zeros((0, 64), device=DEV)), GemmOperand(torch.zeros((8, 64), device=DEV)))
    assert c.shape == (0, 8)
