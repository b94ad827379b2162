"""Dispatch layout at the edges of its two builders: one kernel of 1, 2, 4 or 8 thread blocks for small tables, four kernels
for others; mask words of 32 tokens, blocks without tokens, 1024 experts, unused slots.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2605_05607_b200 import binding as B
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k,G", [(1, 8, 2, 8), (31, 1024, 32, 1024), (256, 8, 8, 1), (257, 12, 3, 4), (513, 6, 1, 3),
                                     (1025, 256, 8, 8), (1100, 64, 4, 32), (4096, 64, 8, 32), (4097, 64, 8, 32),
                                     (16384, 8, 2, 4), (32768, 16, 1, 16), (8192, 128, 4, 8), (8192, 64, 4, 64),
                                     (7000, 256, 4, 256), (12001, 64, 1, 8), (14999, 16, 1, 1),
                                     # dense tables with several mask words per block: the last that the one kernel takes, and beyond
                                     (1777, 128, 4, 8), (2050, 128, 8, 8), (3001, 128, 4, 8), (4096, 64, 8, 8), (4097, 64, 8, 8),
                                     (6441, 128, 4, 8), (6442, 128, 4, 8), (8192, 64, 1, 4), (11366, 64, 1, 4), (11367, 64, 1, 4),
                                     (2900, 256, 4, 64), (2901, 256, 4, 64)])
def test_layout_builders(T, E, k, G):
    rng = np.random.default_rng(T + E)
    skew = -1.5 * np.log(1 + rng.permutation(E))                      # popular and empty experts
    idx = np.argsort(-(rng.gumbel(size=(T, E)) + skew), axis=1)[:, :k].astype(np.int32)
    shape = B.MoEShape(T, 64, 64, E, k, G, 0, 0)
    lay, ws = B.alloc_layout(shape), B.alloc_workspace(shape)
    d_idx = torch.from_numpy(np.ascontiguousarray(idx)).cuda().view(-1)
    for _ in range(2):                                                # the second call finds the first one's scratch
        B.moe_dispatch(shape, None, d_idx, lay, None, ws)
    ref = O.layout(idx, E, G)
    for name in ("expert_counts", "expert_offsets", "group_counts", "group_offsets", "pair_row", "row_pair", "row_src"):
        assert np.array_equal(getattr(lay, name).cpu().numpy()[: ref[name].size], ref[name]), name
    assert np.array_equal(lay.al.cpu().numpy()[: G * T].reshape(G, T), ref["al"])
    assert np.array_equal(lay.disp_token.cpu().numpy()[: ref["n_disp"]], ref["disp_token"])
    pre = B.moe_workspace_layout(shape)["mt_prefix"]
    tiles = np.concatenate([[0], np.cumsum((ref["expert_counts"] + 127) // 128)])
    assert np.array_equal(ws[pre: pre + 4 * (E + 1)].view(torch.int32).cpu().numpy(), tiles)
    assert B.moe_status(ws)[0] == 0


@pytest.mark.parametrize("T", [4096, 4097])
def test_layout_of_a_sparse_table(T):
    """Unused slots (-1): one kernel for 4096 tokens, four for 4097; both against the same layout built slot by slot."""
    E, k = 16, 8
    rng = np.random.default_rng(T)
    idx = np.argsort(rng.random((T, E)), axis=1)[:, :k].astype(np.int32)
    idx[rng.random((T, k)) < 0.8] = -1
    shape = B.MoEShape(T, 64, 64, E, k, 1, 0, B.MOE_FLAG_SPARSE_TOPK)
    lay, ws = B.alloc_layout(shape), B.alloc_workspace(shape)
    B.moe_dispatch(shape, None, torch.from_numpy(idx).cuda().view(-1), lay, None, ws)
    counts = np.bincount(idx[idx >= 0], minlength=E)
    offsets = np.concatenate([[0], np.cumsum(counts)])
    pair_row = np.full(T * k, -1, np.int64)
    flat = idx.reshape(-1)
    for e in range(E):
        pair_row[np.nonzero(flat == e)[0]] = offsets[e] + np.arange(counts[e])      # ascending token
    used = np.nonzero(flat >= 0)[0]
    assert np.array_equal(lay.expert_offsets.cpu().numpy()[: E + 1], offsets)
    assert np.array_equal(lay.pair_row.cpu().numpy()[: T * k], pair_row)
    assert np.array_equal(lay.row_pair.cpu().numpy()[pair_row[used]], used)
    seen = (idx >= 0).any(axis=1)
    assert np.array_equal(lay.al.cpu().numpy()[:T], np.where(seen, np.cumsum(seen) - 1, -1))
    assert np.array_equal(lay.row_src.cpu().numpy()[pair_row[used]], (np.cumsum(seen) - 1)[used // k])
    assert B.moe_status(ws)[0] == 0


@pytest.mark.parametrize("T,E,k,bias", [(1, 8, 2, 0), (32, 32, 32, 0), (33, 33, 5, 33), (256, 64, 4, 0), (257, 128, 8, 128),
                                        (512, 256, 8, 1), (513, 256, 8, 1), (512, 257, 3, 0)])
def test_topk_inside_the_layout_kernel(T, E, k, bias):
    """The layer's routing and layout are those of moe_route and moe_dispatch, whichever kernel takes the top-k."""
    d = f = 64
    g = torch.Generator(device="cuda").manual_seed(T * E)
    x = torch.randn(T, d, generator=g, device="cuda").to(torch.bfloat16)
    wg = torch.randn(d, E, generator=g, device="cuda") * 0.02
    b = None if bias == 0 else torch.randn(*((E,) if bias == 1 else (T, E)), generator=g, device="cuda")
    ws_ = [torch.randn(E, d, f, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]
    shape = B.MoEShape(T, d, f, E, k, 1, T & 1, 0)
    ws, y = B.alloc_workspace(shape), torch.empty(T, d, dtype=torch.bfloat16, device="cuda")
    out = []
    for fused in (False, True):
        logits, idx = torch.empty(T, E, device="cuda"), torch.full((max(T * k, 4),), -7, dtype=torch.int32, device="cuda")
        w, lay = torch.full((max(T * k, 4),), -7.0, device="cuda"), B.alloc_layout(shape)
        if fused:
            B.moe_layer(shape, x, wg, b, *ws_, y, ws, logits=logits, topk_idx=idx, topk_w=w, layout=lay)
        else:
            B.moe_route(shape, x, wg, b, logits, idx, w, ws)
            B.moe_dispatch(shape, None, idx, lay, None, ws)
        out.append((logits, idx, w) + tuple(getattr(lay, n) for n, _ in B.MoELayoutC._fields_))
    for a, c in zip(*out):
        assert torch.equal(a, c)
    assert B.moe_status(ws)[0] == 0


@pytest.mark.parametrize("T,E,k,G", [(32768, 104, 1, 104), (32768, 64, 1, 32), (16384, 128, 2, 128)])
def test_one_token_less_takes_no_longer(T, E, k, G):
    """Whichever builder a table gets, it takes no longer than that of one token more, which has more than 32768 pairs and so
    always the four kernels."""
    def call(T):
        idx = torch.stack([torch.randperm(E, device="cuda")[:k] for _ in range(64)]).to(torch.int32).repeat(T // 64 + 1, 1)[:T]
        idx = idx.contiguous().view(-1)
        shape = B.MoEShape(T, 64, 64, E, k, G, 0, 0)
        lay, ws = B.alloc_layout(shape), B.alloc_workspace(shape)
        return lambda: B.moe_dispatch(shape, None, idx, lay, None, ws)

    us, other = H.device_us(call(T), call(T + 1))
    assert us <= 1.3 * other      # spread of the clock, of a few microseconds
