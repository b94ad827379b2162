"""CPU-side checks of the C-ABI boundary: the library loads, exports every symbol the header
declares, sizes its workspace sensibly and rejects bad arguments before touching a device."""
import ctypes
import functools
import os
import re
import subprocess

import pytest
import torch

from paper_2605_05607_b200 import binding as B
from paper_2605_05607_b200 import build, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build_library()
    return B.lib()


def header_symbols():
    text = open(os.path.join(ROOT, "include", "tcmoe.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(moe_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol(lib):
    names = header_symbols()
    assert set(names) == set(B.EXPORTS), (names, B.EXPORTS)
    for n in names:
        assert getattr(lib, n) is not None


def test_strerror(lib):
    assert B.strerror(0) == "ok"
    assert "workspace" in B.strerror(B.MOE_ERR_WORKSPACE_TOO_SMALL)
    assert "unknown" in B.strerror(12345)


def test_workspace_bytes_and_layout(lib):
    for name, cfg in synth.CONFIGS.items():
        shape = B.make_shape(cfg)
        n = B.moe_workspace_bytes(shape)
        lay = B.moe_workspace_layout(shape)
        P = cfg.T * cfg.k
        assert n >= P * cfg.f * 2 + P * cfg.d * 2            # h and o live inside
        assert lay["status"] == 0 and lay["h"] % 1024 == 0 and lay["o"] % 1024 == 0
        assert lay["o"] - lay["h"] >= P * cfg.f * 2
        assert n < 8e9, name


@pytest.mark.parametrize("kw,code", [
    (dict(k=9), B.MOE_ERR_INVALID_ARG),            # k > E
    (dict(G=3), B.MOE_ERR_INVALID_ARG),            # E % G != 0
    (dict(T=-1), B.MOE_ERR_INVALID_ARG),
    (dict(score_fn=2), B.MOE_ERR_INVALID_ARG),
    (dict(d=100), B.MOE_ERR_UNSUPPORTED_SHAPE),    # d % 8 != 0
    (dict(f=12), B.MOE_ERR_UNSUPPORTED_SHAPE),
    (dict(E=2048, G=8, k=2), B.MOE_ERR_UNSUPPORTED_SHAPE),
    (dict(E=64, k=33, G=8), B.MOE_ERR_UNSUPPORTED_SHAPE),
    (dict(T=2 ** 30, k=2), B.MOE_ERR_UNSUPPORTED_SHAPE),
])
def test_bad_shapes_rejected(lib, kw, code):
    cfg = synth.CONFIGS["C1"].with_(**kw)
    with pytest.raises(B.MoEError) as ei:
        B.moe_workspace_bytes(B.make_shape(cfg))
    assert ei.value.code == code


def test_bad_flags_rejected(lib):
    with pytest.raises(B.MoEError) as ei:
        B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"], flags=1 << 12))
    assert ei.value.code == B.MOE_ERR_INVALID_ARG
    with pytest.raises(B.MoEError) as ei:   # the two forced GEMM-2 forms exclude each other
        B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"], flags=B.MOE_FLAG_GEMM2_PAIR | B.MOE_FLAG_GEMM2_SINGLE))
    assert ei.value.code == B.MOE_ERR_INVALID_ARG
    # the weight cannot be applied in Combine when Combine happens inside GEMM-2's epilogue
    with pytest.raises(B.MoEError) as ei:
        B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"], flags=3))
    assert ei.value.code == B.MOE_ERR_INVALID_ARG
    for bad in (128 | 8, 128 | 512, 256, 16):            # pair GEMM-1 inside the tracker kernel / with its opposite; options without their base flag
        with pytest.raises(B.MoEError):
            B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"], flags=bad))
    for ok in (0, 1, 2, 4, 5, 8, 9, 24, 32, 64, 128, 512, 8 | 256, 8 | 16 | 256):
        assert B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"], flags=ok)) > 0
    # the Mixtral-shaped layer takes the CTA-pair GEMM-1 by itself: its workspace holds the per-expert layout tensors
    c2 = synth.CONFIGS["C2"]
    assert (B.moe_workspace_bytes(B.make_shape(c2)) - B.moe_workspace_bytes(B.make_shape(c2, B.MOE_FLAG_GEMM1_GATHER))
            >= c2.P * c2.d * 2)
    # k = 1: the fp32 token accumulators are larger than o and the workspace accounts for them
    c = synth.CONFIGS["C1"].with_(k=1)
    assert B.moe_workspace_bytes(B.make_shape(c)) >= c.T * c.d * 4 + c.T * c.f * 2


def test_argument_checks_happen_before_any_device_work(lib):
    """Null / misaligned pointers and a short workspace are rejected on the host; with valid
    arguments but no GPU the call reports MOE_ERR_CUDA instead of falling back to anything."""
    cfg = synth.CONFIGS["C1"].with_(T=8)
    shape = B.make_shape(cfg)
    n = B.moe_workspace_bytes(shape)
    ws = torch.zeros(n + 256, dtype=torch.uint8)
    base = ws.data_ptr()
    pad = (-base) % 128
    ws_al = ws[pad: pad + n]
    f32 = torch.zeros(cfg.T * cfg.E, dtype=torch.float32)
    i32 = torch.zeros(cfg.T * cfg.k, dtype=torch.int32)
    w = torch.zeros(cfg.T * cfg.k, dtype=torch.float32)

    def rc(fn):
        try:
            fn()
        except B.MoEError as e:
            return e.code
        return 0

    # null outputs
    assert rc(lambda: B.moe_route(shape, None, None, None, None, i32, w, ws_al)) == B.MOE_ERR_INVALID_ARG
    # workspace too small
    assert rc(lambda: B.moe_route(shape, None, None, None, f32, i32, w, ws_al[:1024])) == B.MOE_ERR_WORKSPACE_TOO_SMALL
    # misaligned workspace
    assert rc(lambda: B.moe_route(shape, None, None, None, f32, i32, w, ws[pad + 4: pad + 4 + n])) == B.MOE_ERR_MISALIGNED
    # bias stride must be 0 or E
    lib_rc = B.lib().moe_route(ctypes.byref(shape), None, None, f32.data_ptr(), 3, f32.data_ptr(), i32.data_ptr(),
                               w.data_ptr(), ws_al.data_ptr(), n, None)
    assert lib_rc == B.MOE_ERR_INVALID_ARG
    # null layout
    assert B.lib().moe_dispatch(ctypes.byref(shape), None, i32.data_ptr(), None, None, ws_al.data_ptr(), n,
                                None) == B.MOE_ERR_INVALID_ARG
    # gate gradient: sigmoid scores need the forward's logits; a short backward workspace is refused
    lay = B.Layout(**{k: torch.zeros(64, dtype=torch.int32) for k in ("expert_counts", "expert_offsets", "group_counts",
                                                                      "group_offsets", "pair_row", "row_pair", "al",
                                                                      "disp_token", "row_src")})
    nb = B.moe_backward_workspace_bytes(shape)
    bws = torch.zeros(nb + 256, dtype=torch.uint8)
    bws_al = bws[(-bws.data_ptr()) % 128:][:nb]
    dxb = torch.zeros(cfg.T * cfg.d * 2 + 256, dtype=torch.uint8)
    dx = dxb[(-dxb.data_ptr()) % 128:][: cfg.T * cfg.d * 2]
    wg = torch.zeros(cfg.d * cfg.E, dtype=torch.float32)
    sig = B.make_shape(cfg.with_(score_fn=1))
    assert rc(lambda: B.moe_gate_backward(sig, None, None, i32, w, lay, wg, dx, wg.clone(), bws_al)) == B.MOE_ERR_INVALID_ARG
    assert rc(lambda: B.moe_gate_backward(shape, None, None, i32, w, lay, wg, dx, wg.clone(), bws_al[:4096])) \
        == B.MOE_ERR_WORKSPACE_TOO_SMALL
    assert rc(lambda: B.moe_gate_backward(B.make_shape(cfg, B.MOE_FLAG_FUSED_FFN), None, None, i32, w, lay, wg, dx,
                                          wg.clone(), bws_al)) == B.MOE_ERR_INVALID_ARG
    if not torch.cuda.is_available():
        assert rc(lambda: B.moe_route(shape, None, None, None, f32, i32, w, ws_al)) == B.MOE_ERR_CUDA
        assert rc(lambda: B.moe_status(ws_al)) == B.MOE_ERR_CUDA
        assert rc(lambda: B.moe_gate_backward(shape, None, None, i32, w, lay, wg, dx, wg.clone(), bws_al)) == B.MOE_ERR_CUDA


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(B, "_lib_handle", None)
    monkeypatch.setattr(B, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        B.moe_workspace_bytes(B.make_shape(synth.CONFIGS["C1"]))


def test_payload_efficiency_matches_the_oracle_and_the_printed_pair(lib):
    """Host-only entry point: the same flit counts as the oracle's packet model on a sweep of sizes and target
    counts, the paper's printed 80 % -> 69 % (Sec. III-A) at eight targets, bad arguments refused."""
    from oracle import moe_oracle as O
    for nbytes in (1, 16, 17, 128, 256, 257, 640, 1280, 4096, 2 * 7168, 2 * 2880):
        for n in (0, 1, 7, 8, 9, 16, 32):
            got, ref = B.moe_payload_efficiency(nbytes, n), O.payload_efficiency(nbytes, n)
            assert got == ref, (nbytes, n, got, ref)
    r = B.moe_payload_efficiency(1280, 8)
    assert round(r["ideal"], 2) == 0.80 and round(r["explicit"], 2) == 0.69 and r["explicit"] < r["dynamic"] < r["ideal"]
    for bad in ((0, 8), (-5, 1), (256, -1), (256, 1 << 15)):
        with pytest.raises(B.MoEError):
            B.moe_payload_efficiency(*bad)


CSRC = os.path.join(ROOT, "paper_2605_05607_b200", "csrc")


@functools.lru_cache(None)
def source(fn):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())


def body_at(text, start):
    """The brace block that opens at or behind `start`."""
    start = text.index("{", start)
    depth, i = 0, start
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
        i += 1


def kernels():
    for fn in sorted(os.listdir(CSRC)):
        if fn.endswith((".cu", ".cuh")):
            text = source(fn)
            for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\(", text):
                depth, i = 1, m.end()
                while depth:
                    depth += {"(": 1, ")": -1}.get(text[i], 0)
                    i += 1
                yield fn, m.group(1), text[m.end():i - 1], body_at(text, i)


@functools.lru_cache(None)
def pointer_fields(kind):
    for fn in sorted(os.listdir(CSRC)):
        m = re.search(rf"\bstruct {kind} \{{", source(fn)) if fn.endswith((".cu", ".cuh")) else None
        if m:
            return re.findall(r"\*\s*(\w+)", body_at(source(fn), m.start()))
    return []


WAIT = "grid_dependency_sync();"
# The kernels that may wait later than at their start, and the condition under which the others of their forms wait there
EARLY = {"ffn_gemm1_kernel": "if (!PLAIN)", "combine_kernel": "if (!EARLY)"}
# What GEMM-2 and Combine share with the kernel before them, or read beside it: not before the wait
GEMM2_ROWS = r"\bp\.(a_src|a_scale|gather_idx|out|topk_w|row_pair|b_scale|b_scale2|y_acc)\b"
COMBINE_ROWS = r"\bc\.(o|y|pg)\b"


def test_every_kernel_waits_for_its_stream_predecessor():
    """All kernels are launched so that they may start while the kernel before them still runs.  Each has to wait for it before it touches
    global memory, with two exceptions that read tables and weights earlier (the tests below), and on every path: the wait also
    completes the chain for the kernel after it."""
    seen = 0
    for fn, name, params, body in kernels():
        pre, found, _ = body.partition(WAIT)
        assert found, f"{fn}: {name} never waits"
        guard = re.split(r"[;{}]", pre)[-1].strip()
        assert guard == EARLY.get(name, ""), f"{fn}: {name} waits under {guard!r}"
        assert pre.count("{") - pre.count("}") == 1, f"{fn}: {name} waits inside a block"
        pointers = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)", params)
        for used in pointers:
            assert not re.search(rf"\b{used}\b", pre), f"{fn}: {name} uses {used} before it waits"
        for kind, v in re.findall(r"\b([A-Z]\w+)\s+(\w+)\s*(?:,|$)", params):
            for field in pointer_fields(kind):
                assert not re.search(rf"\b{v}\.{field}\b", pre), f"{fn}: {name} uses {v}.{field} before it waits"
        assert not re.search(r"__ld|atomic|tma_load|cp_async", pre), f"{fn}: {name}"
        seen += 1
    assert seen >= 25
    # dependents are let go by the wait alone, behind it
    triggers = [fn for fn in os.listdir(CSRC) if fn.endswith((".cu", ".cuh")) and "launch_dependents" in source(fn)]
    text = source("common.cuh")
    assert triggers == ["common.cuh"] and text.count("launch_dependents") == 1
    assert text.index("griddepcontrol.wait") < text.index("griddepcontrol.launch_dependents") < text.index("griddepcontrol.wait") + 120


def test_gemm2_touches_rows_only_behind_its_wait():
    """GEMM-2 on single CTAs reads its tables, the abort word and weights beside the kernel before it.  All of them are older than that kernel,
    as long as that kernel lets dependents go behind its own wait (the test above) and writes none of them: only GEMM-1 and
    the quantisation of its output stand before GEMM-2."""
    body = next(b for _, name, _, b in kernels() if name == "ffn_gemm1_kernel")
    shared, roles = body.split("  if (warp < EPI_WARPS) {", 1)
    assert not re.search(GEMM2_ROWS, shared)
    epilogue, rest = roles.split("  } else if (warp == TMA_WARP) {", 1)
    tma, rest = rest.split("  } else if (warp == MMA_WARP) {", 1)
    mma, gather = rest.split("\n  } else {\n", 1)
    for part in (epilogue, gather):
        pre, found, _ = part.partition("if (PLAIN) " + WAIT)
        assert found and not re.search(GEMM2_ROWS, pre) and "{" not in pre
    for part in (tma, mma):
        assert not re.search(GEMM2_ROWS, part)
    text = source("ffn.cu")
    for fn in ("launch_expert_ffn", "launch_expert_ffn_fp8"):
        launches = re.findall(r"\b(launch_\w+|cudaMem\w+)\(", body_at(text, re.search(rf"cudaError_t {fn}\(", text).end()))
        assert launches.count("launch_gemm2_single") == 1
        before = launches[: launches.index("launch_gemm2_single")]
        assert before[-1] == ("launch_quantize_rows" if fn.endswith("fp8") else "launch_gemm1") and "launch_gemm1" in before, before
        assert all("launch_gemm2_single" not in source(f) for f in ("api.cu", "bwd.cu", "ep.cu", "layout.cu"))


def test_combine_touches_rows_only_behind_its_wait():
    """Combine orders its slots beside the GEMM that writes its rows.  The tables are older than that GEMM in one place, the layer, where
    the experts' launches stand directly before it; there alone it is told that it may."""
    kernel = next(b for _, name, _, b in kernels() if name == "combine_kernel")
    assert not re.search(COMBINE_ROWS, kernel) and kernel.rstrip("} \n").endswith("if (EARLY) " + WAIT)
    token = body_at(source("combine.cuh"), source("combine.cuh").index("void combine_token("))
    pre, found, rows = token.partition("if (EARLY) " + WAIT)
    assert found and not re.search(COMBINE_ROWS, pre) and "combine_rows<" not in pre and "combine_two<" not in pre
    calls = [(fn, m) for fn in os.listdir(CSRC) if fn.endswith(".cu")
             for m in re.finditer(r"[^;]*;[^;]*\blaunch_combine(?:_rows)?\([^;]*, true\)\)?;", source(fn))]
    assert [fn for fn, _ in calls] == ["api.cu"]
    before, call = calls[0][1].group(0).split(";")[:2]
    assert re.search(r"launch_expert_ffn_fp8\(s, a, q, st\) : launch_expert_ffn\(s, a, st\)\)$", before) and "launch_combine(" in call
    assert "bool early = false" in source("common.cuh")


def test_every_tensor_memory_load_is_waited_for_by_name():
    """tcgen05.ld fills its registers some time after it was issued.  Only a wait that has the registers as operands keeps their uses
    below it, so every array that is loaded has to be named by a wait before the next line that is neither load nor wait."""
    csrc = os.path.join(ROOT, "paper_2605_05607_b200", "csrc")
    assert not re.search(r"tcgen05\.wait::ld[^;]*;\"\s*:::", open(os.path.join(csrc, "ptx.cuh")).read())
    seen = 0
    for fn in sorted(os.listdir(csrc)):
        if not fn.endswith(".cu"):
            continue
        pending = set()
        for line in open(os.path.join(csrc, fn)):
            code = line.split("//")[0].strip()
            load, wait = re.search(r"tmem_ld\d+\(.*, (\w+)\);", code), re.search(r"tmem_ld_wait_on\(([^)]*)\);", code)
            if load:
                pending.add(load.group(1))
                seen += 1
            elif wait:
                pending -= set(wait.group(1).replace(" ", "").split(","))
            elif code and not code.startswith(("#pragma", "for (int t = 1; t < 3")):
                assert not pending, f"{fn}: {pending} used before a wait that names them: {code}"


def test_gate_gradient_finds_its_slot_at_the_largest_shapes(tmp_path):
    """The lanes of a token are k rounded up to a power of two, so an accepted shape (T k < 2^31) has up to nearly 2^32 of them.  The lines of
    the kernel that turn a thread into its token and slot, compiled for the CPU, at the ends of the first, a middle and the last token."""
    text = open(os.path.join(ROOT, "paper_2605_05607_b200", "csrc", "gate_bwd.cu")).read()
    body = text[text.index("gate_route_bwd_kernel("):]
    lines = re.search(r"grid_dependency_sync\(\);\n(.*?)\n  const bool slot = ([^;]*);", body, re.S)
    scale = re.search(r"int (shift|width)\) \{", body).group(1)           # what the kernel is told of the lanes per token
    src = tmp_path / "slot.cpp"
    src.write_text("struct Dim { unsigned x; };\n"
                   f"extern \"C\" int slot_of(unsigned block, unsigned threads, unsigned thread, int T, int k, int {scale}, long long* out) {{\n"
                   "  const Dim blockIdx{block}, blockDim{threads}, threadIdx{thread};\n"
                   f"{lines.group(1)}\n  out[0] = t;\n  out[1] = j;\n  return {lines.group(2)};\n}}\n")
    subprocess.run(["g++", "-shared", "-fPIC", "-fwrapv", "-o", str(tmp_path / "slot.so"), str(src)], check=True)
    fn = ctypes.CDLL(str(tmp_path / "slot.so")).slot_of
    out = (ctypes.c_longlong * 2)()
    for k in (1, 2, 3, 8, 9, 16, 17, 31, 32):
        T, shift = (2 ** 31 - 1) // k, (k - 1).bit_length()
        for t in (0, T // 2, T - 1, T):
            for j in (0, k - 1, (1 << shift) - 1):
                block, thread = divmod((t << shift) + j, 256)
                inside = fn(block, 256, thread, T, k, shift if scale == "shift" else 1 << shift, out)
                assert tuple(out) == (t, j) and bool(inside) == (t < T and j < k), (T, k, t, j, tuple(out))


def enclosing_blocks(text, at):
    """(line up to the brace, body start, body end) of the brace blocks around offset `at`, outermost first."""
    out, opened = [], []
    for i, c in enumerate(text):
        if c == "{":
            opened.append(i)
        elif c == "}":
            start = opened.pop()
            if start < at < i:
                out.append((text[text.rfind("\n", 0, start) + 1:start], start, i))
    return out[::-1]


def test_warps_that_meet_inside_a_loop_do_not_leave_it():
    """A barrier of some of a block's warps never completes once one of them has left.  Whether a warp's bounded wait ends with its tile or
    with an abort is a race between the warps, so in a loop with such barriers neither the head nor the body may end it early: in the form of a
    kernel that has the barriers (TILE_OUT) every warp walks every tile."""
    seen = 0
    for fn in sorted(os.listdir(CSRC)):
        if not fn.endswith(".cu"):
            continue
        text = source(fn)
        for m in re.finditer(r"ptx::named_barrier\(|\bfree_boxes\(\)", text):
            loops = [b for b in enclosing_blocks(text, m.start()) if re.search(r"\b(for|while) \(", b[0])]
            if not loops and re.search(r"auto free_boxes = \[&\] \{[^}]*$", text[: m.start()]):
                continue                                                # the helper's own; its calls are looked at
            assert loops, f"{fn}: a named barrier outside of a loop"
            head, start, end = loops[0]
            assert "abort" not in head.replace("(TILE_OUT || !*abort_flag)", ""), f"{fn}: {head.strip()}"
            body = text[start:end].replace("if (!TILE_OUT && !go) break;", "")
            for leave in re.finditer(r"\b(break|return|goto|continue)\b[^;]*;", body):
                own = re.search(r"\[&\]\([^)]*\) \{[^}]*$", body[: leave.start()])   # a lambda's own return
                assert own, f"{fn}: {body[leave.start() - 60:leave.end()]}"
            seen += 1
    assert seen >= 5


def test_product_package_never_imports_the_oracle():
    pkg = os.path.join(ROOT, "paper_2605_05607_b200")
    pat = re.compile(r"^\s*(from|import)\s+oracle\b|oracle[/.]moe_oracle|#include\s+\".*oracle", re.M)
    for dirpath, _, files in os.walk(pkg):
        for fn in files:
            if fn.endswith((".py", ".cu", ".cuh", ".h")):
                assert not pat.search(open(os.path.join(dirpath, fn)).read()), fn


def test_seeded_inputs_are_reproducible_and_independent_per_tensor():
    """The same configuration gives the same bits; changing one shape parameter reshuffles only the
    tensors whose shape depends on it (one generator sub-stream per tensor)."""
    cfg = synth.CONFIGS["C1"].with_(T=64)
    a = {n: synth.tensor_checksum(v) for n, v in synth.make_inputs(cfg).items()}
    b = {n: synth.tensor_checksum(v) for n, v in synth.make_inputs(cfg).items()}
    assert a == b and a["x"] is not None and a["bias"] is None
    c = {n: synth.tensor_checksum(v) for n, v in synth.make_inputs(cfg.with_(T=32)).items()}
    assert c["x"] != a["x"] and all(c[n] == a[n] for n in ("w_gate", "w1", "w3", "w2"))
    d = {n: synth.tensor_checksum(v) for n, v in synth.make_inputs(cfg.with_(seed=1)).items()}
    assert all(d[n] != a[n] for n in ("x", "w_gate", "w1", "w3", "w2"))
