"""moe_launch_count: what the entry points launch, by the forms they take."""
import pytest
import torch

from paper_2605_05607_b200 import binding as B
from paper_2605_05607_b200 import synth

pytestmark = pytest.mark.gpu


def launches(call):
    before = B.moe_launch_count()
    call()
    return B.moe_launch_count() - before


@pytest.mark.parametrize("T,fp8,n", [(64, False, 5), (64, True, 7), (600, False, 6), (20000, False, 9)])
def test_launches_of_a_layer(T, fp8, n):
    """gate, top-k and layout (one kernel for a small batch, two, or five for many pairs), two GEMMs, combine; 8 bits: the quantisation
    of x and of h besides."""
    cfg = synth.MoEConfig("launches", T=T, d=512, f=512, E=8, k=2, G=1)
    t = synth.make_inputs(cfg, "cuda")
    shape = B.make_shape(cfg)
    ws, y = B.alloc_workspace(shape), torch.empty(T, cfg.d, dtype=torch.bfloat16, device="cuda")
    if not fp8:
        assert launches(lambda: B.moe_layer(shape, t["x"], t["w_gate"], None, t["w1"], t["w3"], t["w2"], y, ws)) == n
        return
    q = []
    for name in ("w1", "w3", "w2"):
        E, K, N = t[name].shape
        q += [torch.empty(E, N, K, dtype=torch.uint8, device="cuda"), torch.empty(E, N, device="cuda")]
        assert launches(lambda: B.moe_quantize_weights(t[name], *q[-2:])) >= 1
    assert launches(lambda: B.moe_layer_fp8(shape, t["x"], t["w_gate"], None, *q, y, ws)) == n


@pytest.mark.parametrize("T,kernel", [(512, "topk_layout"), (600, "topk")])
def test_brackets_of_the_topk(T, kernel):
    """The kernel that takes the top-k and the layout of a small batch together has a bracket of its own."""
    cfg = synth.MoEConfig("brackets", T=T, d=512, f=512, E=8, k=2, G=1)
    t = synth.make_inputs(cfg, "cuda")
    shape = B.make_shape(cfg)
    ws, y = B.alloc_workspace(shape), torch.empty(T, cfg.d, dtype=torch.bfloat16, device="cuda")
    for name in ("topk", "topk_layout"):
        B.moe_profile_enable(B.KERNEL_IDS[name])
        B.moe_layer(shape, t["x"], t["w_gate"], None, t["w1"], t["w3"], t["w2"], y, ws)
        ms, n = B.moe_profile_read()
        B.moe_profile_enable(0)
        assert n == (name == kernel) and (ms > 0) == (n > 0), name
