"""GELU and gated GELU of bf16 inputs by the table of the tail erfc(|h| / sqrt 2): the codes of the per-element evaluation, byte for
byte, on every bf16 bit pattern (infinities, NaNs, subnormals among them), behind ordinary, tiny and huge scales."""
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
