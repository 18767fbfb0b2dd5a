"""Quantizer variants chosen by size.  GELU and gated GELU of bf16 inputs by the table of the tail erfc(|h| / sqrt 2): the codes of the per-element evaluation, byte for
byte, on every bf16 bit pattern (infinities, NaNs, subnormals among them), behind ordinary, tiny and huge
scales; and small inputs, four elements a thread, against the same rows of an input that threads of sixteen walk."""
import pytest
import torch

from paper_2507_14811_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def by_mode(mode, *args):
    B.segquant_set_quantize_tuning(mode)
    try:
        return B.segquant_quantize_act_fused(*args)
    finally:
        B.segquant_set_quantize_tuning(0)


@pytest.mark.parametrize("act", ["gelu", "geglu"])
@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True), ("e4m3", False)])
@pytest.mark.parametrize("M,K,kb,scale,mult", [
    # one chunk per row; rows that end between blocks, several K-segments; many rows per thread; scales outside the fast form
    (4096, 16, [0, 16], 0.02, False), (333, 208, [0, 96, 208], 0.02, True), (9001, 304, [0, 304], 0.05, False),
    (300, 256, [0, 256], 1e-30, False), (300, 256, [0, 256], 1e32, True),
])
def test_table_equals_the_per_element_evaluation(act, code, dual, M, K, kb, scale, mult):
    g = torch.Generator().manual_seed(M + K)
    H = (torch.randn((M, K * (2 if act == "geglu" else 1)), generator=g) * 2.5).to(torch.bfloat16)
    bits = torch.arange(65536, dtype=torch.int32).to(torch.int16).view(torch.bfloat16)
    gate = H[:, -K:].reshape(-1)
    gate[: min(65536, gate.numel())] = bits[: gate.numel()]
    H[:, -K:] = gate.view(M, K)
    sp = torch.full((len(kb) - 1,), scale, device=DEV)
    args = (H.to(DEV), B.SegTable(kb, [0, 64]), sp, sp * 0.5 if dual else None, code, act,
            (torch.rand(K, generator=g) + 0.5).to(DEV) if mult else None)
    for want, got in zip(by_mode(2, *args), by_mode(1, *args)):
        assert (want is None and got is None) or torch.equal(want, got)


@pytest.mark.parametrize("act,K", [(None, 1043), ("silu", 1043), ("gelu", 1042), ("geglu", 1048)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True), ("e4m3", False)])
def test_small_inputs_equal_rows_of_a_large_one(act, K, dtype, code, dual):
    """Row tails and segment bounds that cut a thread's four elements, and a scale outside the fast form in one segment."""
    g = torch.Generator(device=DEV).manual_seed(K)
    kb, M = [0, 33, 514, K], 6000
    H = torch.zeros((M, 2 * 1056), dtype=dtype, device=DEV)[:, : 2 * K if act == "geglu" else K]
    H.copy_(torch.randn(H.shape, generator=g, device=DEV) * 2.0)
    sp = torch.tensor([0.02, 0.03, 2.0 ** -90], device=DEV)
    mult = torch.rand(K, generator=g, device=DEV) + 0.5 if act else None
    run = lambda rows: B.segquant_quantize_act_fused(H[rows], B.SegTable(kb, [0, 8]), sp, sp * 0.5 if dual else None, code, act, mult)
    whole = run(slice(0, M))
    for rows in (slice(0, 1), slice(2995, 3000), slice(M - 130, M)):
        for w, p in zip(whole, run(rows)):
            assert (w is None and p is None) or torch.equal(w[rows], p)


def test_small_zero_point_inputs_equal_rows_of_a_large_one():
    g = torch.Generator(device=DEV).manual_seed(3)
    X = torch.randn((6000, 1056), generator=g, device=DEV, dtype=torch.float32)[:, :1043]
    seg = B.SegTable([0, 33, 1043], [0, 8])
    s_x, z_x = torch.tensor([0.02, 0.03], device=DEV), torch.tensor([-7, 100], dtype=torch.int32, device=DEV)
    whole = B.segquant_quantize_act_zero_point(X, seg, s_x, z_x)
    assert torch.equal(whole[40:47], B.segquant_quantize_act_zero_point(X[40:47], seg, s_x, z_x))


@pytest.mark.parametrize("N,K", [(1, 16), (7, 48), (257, 4112), (3100, 4096), (2049, 7984)])
def test_packed_codes_come_back(N, K):
    """One and several chunks per thread, grids that the chunks do not fill, a row pitch wider than the row."""
    g = torch.Generator(device=DEV).manual_seed(N)
    codes = torch.randint(-8, 8, (N, K), generator=g, device=DEV, dtype=torch.int8)
    w8 = B.new_codes(N, K, DEV)
    w8.copy_(codes.view(torch.uint8))
    w4 = B.segquant_pack_w4(w8)
    low, high = codes[:, 0::2].to(torch.int32) & 15, codes[:, 1::2].to(torch.int32) & 15
    assert torch.equal(w4.to(torch.int32), low | high << 4)
    out = torch.full((N + 1, w8.stride(0)), 77, dtype=torch.uint8, device=DEV)
    B.segquant_unpack_w4(w4, out=out[:N, :K])
    assert torch.equal(out[:N, :K], codes.view(torch.uint8))
    assert bool(torch.all(out[:N, K:] == 77)) and bool(torch.all(out[N] == 77))


@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True), ("e4m3", False)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("M,kb", [(40, [0, 520, 1056]), (6000, [0, 520, 1056]), (6000, [0, 512, 1056])])
def test_infinities_saturate(M, kb, dtype, code, dual):
    """Infinite inputs, and infinities that a gated product or a multiplier makes of finite ones, get the ends of the code
    range: in whole chunks and in those that a segment bound cuts, with few and many elements a thread, by table."""
    K = kb[-1]
    big = torch.finfo(dtype).max
    g = torch.Generator(device=DEV).manual_seed(M)
    x = torch.randn((M, K), generator=g, device=DEV)
    pick = torch.randint(0, 8, (M, K), generator=g, device=DEV)
    seg = B.SegTable(kb, [0, 8])
    sp = torch.tensor([0.02, 0.03], device=DEV)
    sn = sp * 0.5 if dual else None
    put = lambda t, v: torch.where(pick == 0, v, torch.where(pick == 1, -v, t)).to(dtype)
    ends = (0x7F, 0x80 if dual else 0x81) if code == "int8" else (0x7E, 0xFE)

    def check(codes):
        for at, pos, neg in ((pick == 0, ends[0], 0), (pick == 1, 0 if dual else ends[1], ends[1])):
            assert bool(torch.all(codes[0][at] == pos)) and (not dual or bool(torch.all(codes[1][at] == neg)))

    check(B.segquant_quantize_act(put(x, float("inf")), seg, sp, sn, code))
    check(B.segquant_quantize_act_fused(put(x, big), seg, sp, sn, code, None, torch.full((K,), 4.0, device=DEV)))
    gated = torch.cat([put(x, big), put(x, 8.0).abs()], 1)               # GELU(8) = 8: the product overflows
    for mode in (1, 2):
        check(by_mode(mode, gated, seg, sp, sn, code, "geglu"))
    if code == "int8" and dual:
        fused = put(x, big).abs()                                        # (no pre-activation has a large negative SiLU or GELU)
        for act in ("silu", "gelu"):
            for mode in (1, 2):
                c_pos, c_neg = by_mode(mode, fused, seg, sp, sn, code, act, torch.full((K,), 4.0, device=DEV))
                assert bool(torch.all(c_pos[pick < 2] == 0x7F)) and bool(torch.all(c_neg[pick < 2] == 0))
