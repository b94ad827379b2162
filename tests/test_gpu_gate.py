"""Gate logits at the edges of the kernel's tiles (128 tokens, 32 / 64 / 128 experts, one or two row tiles, k-blocks of 64,
fewer than 128 rows loaded), against the product in fp64."""
import numpy as np
import pytest
import torch

from paper_2605_05607_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E", [(1, 8, 1), (1, 64, 5), (9, 4096, 8), (127, 520, 64), (128, 7168, 256), (129, 136, 65),
                                   (297, 2880, 128), (2050, 264, 1024), (4097, 72, 160), (20000, 72, 96), (20000, 72, 256)])
def test_gate_logits(T, d, E):
    g = torch.Generator(device="cuda").manual_seed(T + d + E)
    x = torch.randn(T, d, generator=g, device="cuda").to(torch.bfloat16)
    w = torch.randn(d, E, generator=g, device="cuda") * 0.02
    shape = B.MoEShape(T, d, 64, E, 1, 1, 0, 0)
    ws = B.alloc_workspace(shape)
    logits = torch.full((T, E), float("nan"), device="cuda")
    idx = torch.empty(max(T, 4), dtype=torch.int32, device="cuda")
    tw = torch.empty(max(T, 4), device="cuda")
    B.moe_route(shape, x, w, None, logits, idx, tw, ws)
    ref = x.double() @ w.double()
    # every product is exact; 3 d / 16 + 3 additions of partial sums, each off by at most one part in 2^22 of the sum of
    # magnitudes (the tensor pipe truncates)
    bound = (3 * d / 16 + 3) * 2.0 ** -22 * (x.double().abs() @ w.double().abs())
    assert bool(((logits.double() - ref).abs() <= bound).all())
    assert np.array_equal(idx[:T].cpu().numpy(), np.argmax(logits.cpu().numpy(), axis=1))
    # a token's logits do not depend on how many others share the call (other tile forms, the same sums)
    n = min(T, 5)
    few = B.MoEShape(n, d, 64, E, 1, 1, 0, 0)
    logits_few = torch.empty(n, E, device="cuda")
    B.moe_route(few, x[:n].contiguous(), w, None, logits_few, idx, tw, ws)
    assert torch.equal(logits_few, logits[:n]) and B.moe_status(ws)[0] == 0
