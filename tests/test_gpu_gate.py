"""Gate logits at the edges of the kernel's tiles (64 / 128 tokens, 32 / 64 / 128 experts, one or two row tiles, k-blocks of 64,
fewer than 128 rows loaded, weights split inside the GEMM or before it), against the product in fp64."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2605_05607_b200 import binding as B
from tests import helpers as H

# Every form that the library's cost table chooses, with a ragged last row tile, a ragged last column tile and a k-block of 8; two row
# tiles per task with a last task of one tile and with a second tile that is partly filled (the next test checks that they are).
FORM_CASES = [(520, 72, 1001), (1961, 72, 132), (1961, 72, 129), (3140, 72, 132), (3795, 72, 129), (3795, 72, 132),
              (6415, 72, 129), (6284, 72, 132), (9559, 72, 96), (9690, 72, 96), (18991, 72, 33), (4843, 72, 100),
              (9559, 72, 33), (18991, 72, 65), (18991, 72, 96), (6153, 72, 321), (6284, 264, 132), (12572, 72, 129),
              (12703, 72, 132), (511, 72, 161), (512, 72, 164)]
EDGE_CASES = [(1, 8, 1), (1, 64, 5), (9, 4096, 8), (127, 520, 64), (128, 7168, 256), (129, 136, 65), (297, 2880, 128),
              (2050, 264, 1024), (4097, 72, 160), (20000, 72, 96), (20000, 72, 256)]


def test_form_cases_reach_every_form():
    """The cost table is read from the source, so that a new form or a new cost that leaves one uncovered shows here."""
    text = open(os.path.join(os.path.dirname(B.__file__), "csrc", "gate_gemm.cu")).read()
    pre_min = int(re.search(r"PRE_MIN_TOKENS = (\d+);", text).group(1))
    pre_us = float(re.search(r"PRE_US = ([\d.]+);", text).group(1))
    crowd = re.search(r"form\.gn == (\d+) && E > (\d+) && tasks > (\d+) \? ([\d.]+)", text).groups()
    cost = lambda t: None if t == "NO" else tuple(float(v) for v in t.strip("{}").split(","))
    table = [((int(gn), int(bm), int(m), pre == "true"), cost(run), cost(apart)) for gn, bm, m, pre, run, apart in
             re.findall(r"\{\{(\d+), (\d+), (\d+), (true|false)\}, (NO|\{[^}]*\}), (NO|\{[^}]*\})\}", text)]
    assert len(table) == len(re.findall(r"^ *\{\{\d", text, re.M)) >= 8

    def form(T, d, E):
        best = (1e30, None)
        for f, run, apart in table:
            c = apart if E <= 128 else run
            if c is None or (f[3] and T < pre_min):
                continue
            rounds = -(-(-(-T // (f[1] * f[2])) * -(-E // f[0])) // 148)
            us = rounds * (c[0] + -(-d // 64) * c[1 if E % 4 == 0 else 2]) + (pre_us if f[3] else 0.0)
            if f[0] == int(crowd[0]) and E > int(crowd[1]) and -(-T // (f[1] * f[2])) * -(-E // f[0]) > int(crowd[2]):
                us += float(crowd[3])
            best = min(best, (us, f), key=lambda b: b[0])
        return best[1]

    seen = set()
    for T, d, E in FORM_CASES + EDGE_CASES:
        f = form(T, d, E)
        rem = T % (f[1] * f[2])
        if E % f[0] and (rem > f[1] or (rem and f[2] == 1)):
            seen.add((f, E <= 128, "ragged last tile"))
        if f[2] == 2 and E % f[0] and 0 < rem < f[1]:
            seen.add((f, E <= 128, "one row tile in the last task"))
    for f, run, apart in table:
        for c, few in ((run, False), (apart, True)):
            if c is not None:
                assert (f, few, "ragged last tile") in seen, (f, few)
                assert f[2] == 1 or (f, few, "one row tile in the last task") in seen, (f, few)


@pytest.mark.gpu
@pytest.mark.parametrize("T,d,E", EDGE_CASES + FORM_CASES)
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


@pytest.mark.gpu
@pytest.mark.parametrize("T,d,E,wider", [(16384, 2880, 129, 192), (8192, 7168, 250, 256), (16384, 7168, 258, 384),
                                         (16384, 256, 129, 160), (12288, 256, 66, 96)])
def test_fewer_experts_take_no_longer(T, d, E, wider):
    """A number of experts that is no multiple of the tile's width or of 4 costs about what the wider gate costs."""
    def call(E):
        x = torch.randn(T, d, device="cuda").to(torch.bfloat16)
        w = torch.randn(d, E, device="cuda") * 0.02
        shape = B.MoEShape(T, d, 64, E, 1, 1, 0, 0)
        ws = B.alloc_workspace(shape)
        out = torch.empty(T, E, device="cuda"), torch.empty(T, dtype=torch.int32, device="cuda"), torch.empty(T, device="cuda")
        return lambda: B.moe_route(shape, x, w, None, *out, ws)

    # measured, taking turns: 0.99, 1.01, 0.92, 0.98, 0.90; with the split in the GEMM for every size 1.34, 1.68, 1.41 (the first three),
    # with logits stored by the element where E is no multiple of 4 1.45, 1.38 (the last two)
    us, other = H.device_us(call(E), call(wider))
    assert us <= 1.23 * other


@pytest.mark.gpu
@pytest.mark.parametrize("d,E", [(256, 128), (1024, 104)])
def test_a_few_more_row_tiles_take_no_longer(d, E):
    """13 and 16 row tiles of 128 tokens, both at one task per SM: the second call takes what the first does, the top-k of 384 tokens more aside."""
    def call(T):
        x = torch.randn(T, d, device="cuda").to(torch.bfloat16)
        w = torch.randn(d, E, device="cuda") * 0.02
        shape = B.MoEShape(T, d, 64, E, 1, 1, 0, 0)
        ws = B.alloc_workspace(shape)
        out = torch.empty(T, E, device="cuda"), torch.empty(T, dtype=torch.int32, device="cuda"), torch.empty(T, device="cuda")
        return lambda: B.moe_route(shape, x, w, None, *out, ws)

    # measured, taking turns: 1.02, 1.05; in 128 and 112 blocks of 16 columns 1.13, 1.12.  The line lies in the middle.
    us, other = H.device_us(call(2048), call(1664))
    assert us <= 1.08 * other
