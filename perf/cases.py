"""The work that users of this library have it do, as timed cases.

A case is one pass through the public entry points with the buffers that a serving program would hold: tiled weights,
preallocated activations and outputs, a registered workspace.  Shapes are those of ``workloads.py`` (the decoder linears
of the 7B and 13B Llama-2 models, hidden and ffn sizes of which the drawn cases take multiples of 128 in between).

Kinds of case (``kind``):

* ``linear``  one call of one layer, launched directly.
* ``block``   the four linears (``acts`` with act-order: three) of a number of decoder layers, every layer with weights of
              its own.  With ``graph`` the calls are captured once and replayed, as decode loops do; without, they are
              launched one by one, as prefill is.
* ``mlp``     the fused MLP of a block: gate_up with silu(gate) * up in its epilogue, stored in the row order of the
              act-order down projection, which adds bias and residual.
* ``host``    a decode step whose activations live in pinned host memory (gptq_gemm_host_batch).

Options: ``dtype`` fp16 or bf16 (activations, scales, outputs), ``wbits`` 4 or 8, ``group`` (rows per scale; 0 = one
group per column), ``act`` (act-order checkpoint), ``minus_one`` (zero points stored minus one).
"""
from __future__ import annotations

import torch

from paper_2511_19438_b200 import binding as B
from paper_2511_19438_b200 import harness as H
from paper_2511_19438_b200 import workloads as wl

_LAYERS = {"7b": wl.SHAPES_7B, "13b": wl.SHAPES_13B}
_WORKSPACE_BYTES = 256 << 20      # act-order and 8-bit calls gather x here; registered once, like a server does
_MAX_FLOPS = 4 * sum(2 * 1024 * K * N for K, N in wl.SHAPES_7B.values())    # cost bound of a drawn case
_workspace = None


def _case(name, kind, M, **kw):
    c = {"name": name, "kind": kind, "M": M, "model": "7b", "layers": 1, "K": 0, "N": 0, "dtype": "fp16", "wbits": 4,
         "group": 128, "act": False, "minus_one": False, "graph": False}
    c.update(kw)
    return c


def listed():
    return [
        # a single small projection called by itself: what one call costs, host side included
        _case("linear_m1", "linear", 1, K=4096, N=4096),
        # token generation for one user: the linears of eight decoder layers, replayed
        _case("decode7b_m1", "block", 1, layers=8, graph=True),
        # ... for a small and an ordinary batch
        _case("decode7b_m16", "block", 16, layers=8, graph=True),
        _case("decode7b_m64", "block", 64, layers=4, graph=True),
        # act-order checkpoints of the larger model, small batch
        _case("decode13b_actorder_m8", "block", 8, model="13b", layers=4, act=True, graph=True),
        # bfloat16, group size 64, older zero-point convention, an odd batch
        _case("decode7b_bf16_g64_m23", "block", 23, layers=4, dtype="bf16", group=64, minus_one=True, graph=True),
        # the fused MLP of an act-order layer at a handful of sequences
        _case("mlp7b_m5", "mlp", 5, layers=4, act=True, graph=True),
        # a decode step whose activations live on the host
        _case("host7b_m4", "host", 4, layers=8),
        # a large decode batch or a short prompt: no multiple of any tile
        _case("block7b_m100", "block", 100),
        # 8-bit weights, a prompt of a few hundred tokens
        _case("block7b_w8_m300", "block", 300, wbits=8),
        # prompts: one of ordinary length, and a full batch of them
        _case("prefill7b_m512", "block", 512),
        _case("prefill7b_m4096", "block", 4096),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "block", "block", "mlp", "host"])
    wbits = rng.choice([4, 4, 4, 8]) if kind in ("linear", "block", "host") else 4
    dtype = rng.choice(["fp16", "fp16", "bf16"]) if wbits == 4 and kind in ("linear", "block", "host") else "fp16"
    c = _case("", kind, 1, dtype=dtype, wbits=wbits, group=rng.choice([128, 128, 128, 64, 32]), minus_one=rng.random() < 0.2)
    del c["name"]
    if kind == "linear":
        c["K"], c["N"] = 128 * _log_int(rng, 8, 108), 128 * _log_int(rng, 8, 216)
        if rng.random() < 0.15 and wbits == 4:
            c["group"] = 0
        c["act"] = wbits == 4 and c["group"] != 0 and rng.random() < 0.3
        c["M"] = _log_int(rng, 1, 4096)
    elif kind == "block":
        c["model"] = rng.choice(["7b", "13b"])
        c["act"] = rng.random() < 0.3
        c["graph"] = rng.random() < 0.6
        c["M"] = _log_int(rng, 1, 128 if c["graph"] else 4096)
        c["layers"] = rng.choice([2, 3, 4]) if c["M"] <= 128 else 1
    elif kind == "mlp":
        c["model"] = rng.choice(["7b", "13b"])
        c["act"] = True
        c["M"] = _log_int(rng, 1, 64)
        c["layers"], c["graph"] = rng.choice([2, 3, 4]), True
    else:
        c["M"] = _log_int(rng, 1, 64)
        c["layers"] = rng.choice([2, 4, 8])
    while work(c)["flops"] * (c["wbits"] // 4) > _MAX_FLOPS:
        c["M"] = max(1, c["M"] // 2 + c["M"] % 3)
    return c


def _group(case, K):
    return case["group"] or K


def _layer_shapes(case):
    if case["kind"] == "linear":
        return [("linear", (case["K"], case["N"]))]
    shapes = _LAYERS[case["model"]]
    if case["kind"] == "mlp":
        return [(n, shapes[n]) for n in ("gate_up", "down")]
    return list(shapes.items())


def work(case):
    M, nbytes, flops = case["M"], 0, 0
    for name, (K, N) in _layer_shapes(case):
        nbytes += wl.algorithmic_bytes(M, K, N, _group(case, K), case["act"], case["wbits"])
        flops += wl.matmul_flops(M, K, N)
    if case["kind"] == "mlp":
        (_, Ng), (Kd, Nd) = (s for _, s in _layer_shapes(case))
        # silu(gate) * up halves gate_up's output and stays on its way to down (written and read once); residual and bias
        nbytes += -2 * M * Ng + 2 * M * (Ng // 2) + 4 * (Ng // 2) + 2 * M * Nd + 2 * Nd
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * flops}


def tolerance(case):
    # Against the same product in 64 bits the library's outputs show rel 2.1e-4 (up to 16 rows: the one rounding of y) to
    # 2.9e-4 (above: every scaled weight is rounded too) in fp16 and 2.3e-3 in bfloat16; largest differences 4e-3 (one
    # group per column) and 1e-2.  Another implementation of that precision rounds elsewhere: four times as much.
    return {"rel": 1e-2, "max": 4e-2} if case["dtype"] == "bf16" else {"rel": 1.2e-3, "max": 1.6e-2}


def _register_workspace():
    global _workspace
    if _workspace is None:
        _workspace = H.WorkspaceHolder()
    _workspace.ensure(_WORKSPACE_BYTES)


def _make_layer(case, K, N, gen, gate_up=False):
    """A layer with uniform packed words and the scale recipe of ``workloads.make_scales``, repacked."""
    dev, group = "cuda", _group(case, K)
    G, per_word = K // group, 32 // case["wbits"]

    def words(rows, cols):
        return torch.randint(-(1 << 31), 1 << 31, (rows, cols), generator=gen, device=dev, dtype=torch.int64).to(torch.int32)

    qw, qz = words(K // per_word, N), words(G, N // per_word)
    if case["wbits"] == 8:      # a stored byte of 255 has no meaning under the minus-one convention
        qz = qz & 0x7f7f7f7f
    sc = wl.SCALE_FLOOR + (torch.randn((G, N), generator=gen, device=dev) * wl.SCALE_SIGMA).abs()
    sc = sc.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float16)
    gi = None
    if case["act"]:
        gi = (torch.randperm(K, generator=gen, device=dev) // group).to(torch.int32)
    fmt = (B.GPTQ_FORMAT_ZEROS_MINUS_ONE if case["minus_one"] else 0) | (B.GPTQ_FORMAT_GATE_UP if gate_up else 0)
    fmt |= B.GPTQ_FORMAT_BF16 if case["dtype"] == "bf16" else 0
    if case["wbits"] == 8:
        outs = [torch.empty(B.gptq_repack_w8_bytes(w, N, K, group), dtype=torch.uint8, device=dev) for w in range(3)]
        perm = torch.empty(2 * K, dtype=torch.int32, device=dev)
        n = B.gptq_repack_w8_scratch_bytes(N, K, group)
        scratch = torch.empty(n, dtype=torch.uint8, device=dev)
        B.check(B.gptq_repack_w8(qw, qz, sc, gi, *outs, perm, scratch, n, N, K, group, case["act"], fmt), "gptq_repack_w8")
    else:
        outs = [torch.empty(B.gptq_repack_bytes(w, N, K, group, case["act"]), dtype=torch.uint8, device=dev) for w in range(3)]
        perm = torch.empty(K, dtype=torch.int32, device=dev) if case["act"] else None
        B.check(B.gptq_repack_format(qw, qz, sc, gi, *outs, perm, N, K, group, case["act"], fmt), "gptq_repack_format")
    return H.DeviceLinear(K, N, group, case["act"], *outs, perm, None)


def _call(case, op):
    """One library call of a case; ``op`` is what _make_ops laid out."""
    if op["do"] == "silu_mul_scatter":
        H.gemm_silu_mul_scatter(op["x"], op["D"], op["index"], op["y"])
    elif op["do"] == "bias_residual":
        D = op["D"]
        B.check(B.gptq_gemm_bias_residual(op["x"], D.qweight_t, D.qzeros_t, D.scales_t, None, op["bias"], op["residual"],
                                          op["y"], case["M"], D.N, D.K, D.group_size, B.GPTQ_ACT_ORDER_PRESORTED),
                "gptq_gemm_bias_residual")
    elif case["wbits"] == 8:
        H.gemm_w8(op["x"], op["D"], op["y"])
    elif case["dtype"] == "bf16":
        H.gemm_bf16(op["x"], op["D"], op["y"])
    else:
        H.gemm(op["x"], op["D"], op["y"])


def _make_ops(case, gen):
    M, dt = case["M"], torch.bfloat16 if case["dtype"] == "bf16" else torch.float16

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda").to(dt)

    def empty(*shape):
        return torch.empty(shape, dtype=dt, device="cuda")

    ops = []
    for _ in range(case["layers"]):
        if case["kind"] == "mlp":
            (Kg, Ng), (Kd, Nd) = (s for _, s in _layer_shapes(case))
            up = _make_layer(case, Kg, Ng, gen, gate_up=True)
            down = _make_layer(case, Kd, Nd, gen)
            h = empty(M, Ng // 2)
            x = normal(M, Kg)[:, up.perm.long()].contiguous()      # the producer of x wrote it in up's row order
            up.act_order = B.GPTQ_ACT_ORDER_PRESORTED
            ops.append({"do": "silu_mul_scatter", "D": up, "x": x, "index": H.invert_perm(down.perm), "y": h})
            ops.append({"do": "bias_residual", "D": down, "x": h, "bias": normal(Nd), "residual": normal(M, Nd), "y": empty(M, Nd)})
        else:
            for name, (K, N) in _layer_shapes(case):
                ops.append({"do": "gemm", "D": _make_layer(case, K, N, gen), "x": normal(M, K), "y": empty(M, N)})
    return ops


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    _register_workspace()
    ops = _make_ops(case, gen)
    state = {"case": case, "ops": ops, "outputs": [op["y"] for op in ops], "graph": None}
    if case["kind"] == "host":
        items = []
        for op in ops:
            D = op["D"]
            op["x_host"], op["y_host"] = op["x"].cpu().pin_memory(), torch.empty_like(op["y"], device="cpu").pin_memory()
            items.append((op["x_host"], D.qweight_t, D.qzeros_t, D.scales_t, D.perm, op["y_host"], op["x"], op["y"], case["M"],
                          D.N, D.K, D.group_size, case["act"]))
        state["problems"] = B.make_host_problems(items)
        state["outputs"] = [op["y_host"] for op in ops]
    elif case["graph"]:
        for op in ops:
            _call(case, op)
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            for op in ops:
                _call(case, op)
    torch.cuda.synchronize()
    B.check(B.gptq_check_status(), "prepare")
    return state


def run(state):
    case = state["case"]
    if state["graph"] is not None:
        state["graph"].replay()
    elif case["kind"] == "host":
        batch = (B.gptq_gemm_host_batch_w8 if case["wbits"] == 8 else
                 B.gptq_gemm_host_batch_bf16 if case["dtype"] == "bf16" else B.gptq_gemm_host_batch)
        status, bad = batch(state["problems"])
        B.check(status, f"gptq_gemm_host_batch (problem {bad})")
        torch.cuda.current_stream().synchronize()      # the step's results are wanted on the host
    else:
        for op in state["ops"]:
            _call(case, op)
    return state["outputs"]
