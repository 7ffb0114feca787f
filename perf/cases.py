"""What a user of this library has it do, as measurable passes through the public entry points.

A case is a dict of plain values; ``kind`` names the path:

  gemv    one product (bitcos_gemv, trit5_gemv or bit2_gemv), int8 activations with one scale per token
  layer   the seven products of a decoder layer as its four dependent launches (q+k+v, o, gate+up, down);
          ``act`` is what the caller holds: "int8" on the device (bitcos_gemv_multi with the sequence hints),
          "bf16" on the device (bitcos_gemv_multi_bf16: quantised inside the launch), or "host" (HostPhases: pinned
          activations in, pinned outputs back)
  quant   bf16 activations quantised per group of 128, then the product with group scales
  blend   the 16-bit variant: weights +-s against unquantised bf16 activations
  moe     top-k routed experts: pairs grouped on the device, then the gate, up and down products
  pack    dense trits and scales in device memory -> the packed buffers (the set-up path)

Shapes, densities and distributions are those of the library's own configurations (datagen's five), or lie in
the ranges around them; everything is made from the seed with torch generators on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_16338_b200 as bc

GROUP = 128
ROWS = 32


def listed():
    return [
        # the smallest product of the configurations: latency and launch cost only
        {"name": "gemv_256x512_b1", "kind": "gemv", "fmt": "bitcos", "M": 256, "K": 512, "batch": 1, "z": 0.42},
        # an ordinary projection of a mid-sized model, one decode token
        {"name": "gemv_4096x12288_b1", "kind": "gemv", "fmt": "bitcos", "M": 4096, "K": 12288, "batch": 1, "z": 0.42},
        # a tensor so dense that the format choice stores it as five-trit; ragged rows, two tokens
        {"name": "gemv_trit5_12277x4096_b2", "kind": "gemv", "fmt": "trit5", "M": 12277, "K": 4096, "batch": 2, "z": 0.30},
        # one decode token through the layer of a 2B model: four short dependent launches
        {"name": "layer_2b_b1", "kind": "layer", "act": "int8", "hidden": 2560, "q": 2560, "kv": 640, "ffn": 6912, "batch": 1,
         "z": 0.4219},
        # the same from pinned host buffers to pinned host buffers, the whole call
        {"name": "layer_2b_host_b1", "kind": "layer", "act": "host", "hidden": 2560, "q": 2560, "kv": 640, "ffn": 6912, "batch": 1,
         "z": 0.4219},
        # the same for two tokens whose activations are still 16-bit
        {"name": "layer_2b_bf16_b2", "kind": "layer", "act": "bf16", "hidden": 2560, "q": 2560, "kv": 640, "ffn": 6912, "batch": 2,
         "z": 0.4219},
        # one decode token through the layer of a 32B model: the largest packed matrices
        {"name": "layer_32b_b1", "kind": "layer", "act": "int8", "hidden": 5120, "q": 8192, "kv": 1024, "ffn": 25600, "batch": 1,
         "z": 0.4711},
        # the same for the largest batch
        {"name": "layer_32b_b16", "kind": "layer", "act": "int8", "hidden": 5120, "q": 8192, "kv": 1024, "ffn": 25600, "batch": 16,
         "z": 0.4711},
        # the quantised front end as two calls, a small odd batch, ragged rows
        {"name": "quant_2555x6912_b5", "kind": "quant", "M": 2555, "K": 6912, "batch": 5, "z": 0.4219},
        # callers that cannot quantise their activations
        {"name": "blend_8192x5120_b4", "kind": "blend", "M": 8192, "K": 5120, "batch": 4, "z": 0.4711},
        # mixture-of-experts decode with the routing left on the device
        {"name": "moe_128x768x2048_b8", "kind": "moe", "experts": 128, "top_k": 8, "hidden": 2048, "ffn": 768, "batch": 8, "z": 0.3288},
        # packing a projection at load time
        {"name": "pack_8192x5120", "kind": "pack", "M": 8192, "K": 5120, "z": 0.4711},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log_groups(rng, lo, hi):
    return GROUP * _log_int(rng, lo // GROUP, hi // GROUP)


def _shape(rng, most):
    """M of any residue modulo 32 and K a multiple of 128, each over the range the configurations span."""
    while True:
        M, K = _log_int(rng, 64, 25600), _log_groups(rng, 128, 25600)
        if rng.random() < 0.5:
            M = max(ROWS, M // ROWS * ROWS)
        if 1 << 15 <= M * K <= most:
            return M, K


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "gemv", "layer", "layer", "quant", "blend", "moe", "pack"])
    z = round(rng.uniform(0.30, 0.515), 4)
    if kind == "gemv":
        M, K = _shape(rng, 25600 * 5120)
        return {"kind": kind, "fmt": rng.choice(["bitcos", "bitcos", "bitcos", "trit5", "bit2"]), "M": M, "K": K,
                "batch": rng.choice([1, 1, 1, 2, 3, 4, 5, 8, 11, 16]), "z": z}
    if kind == "layer":
        hidden = _log_groups(rng, 1024, 5120)
        act = rng.choice(["int8", "int8", "bf16", "host"])
        return {"kind": kind, "act": act, "hidden": hidden, "q": rng.choice([hidden, _log_groups(rng, 1024, 8192)]),
                "kv": _log_groups(rng, 256, 1024), "ffn": _log_groups(rng, 2 * hidden, 5 * hidden),
                "batch": rng.choice([1, 2]) if act == "bf16" else rng.choice([1, 1, 2, 4, 7, 16]), "z": z}
    if kind == "quant":
        M, K = _shape(rng, 8192 * 5120)
        return {"kind": kind, "M": M, "K": K, "batch": rng.randint(1, 16), "z": z}
    if kind == "blend":
        M, K = _shape(rng, 8192 * 5120)
        return {"kind": kind, "M": M, "K": K, "batch": rng.randint(1, 8), "z": z}
    if kind == "moe":
        return {"kind": kind, "experts": rng.choice([32, 64, 128]), "top_k": rng.choice([4, 8]), "hidden": _log_groups(rng, 1024, 2560),
                "ffn": _log_groups(rng, 384, 1024), "batch": rng.randint(1, 16), "z": z}
    M, K = _shape(rng, 25600 * 5120)
    return {"kind": kind, "M": M, "K": K, "z": z}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _trits(gen, M, K, z):
    """int8 [M, K]: 0 with probability z, else +-1 evenly."""
    u = torch.rand((M, K), generator=gen, device="cuda")
    return (u >= z).to(torch.int8) - 2 * (u >= z + (1.0 - z) / 2.0).to(torch.int8)


def _trits_fixed_count(gen, M, K, z):
    """The same with exactly round(z K) zeros in every row, so that the packed sizes depend on the shape alone."""
    order = torch.rand((M, K), generator=gen, device="cuda").argsort(dim=1)[:, round(z * K):]
    t = torch.zeros((M, K), dtype=torch.int8, device="cuda")
    return t.scatter_(1, order, (2 * torch.randint(0, 2, order.shape, generator=gen, device="cuda", dtype=torch.int8) - 1))


def _scales(gen, M, K):
    """bf16 scales U[0.01, 0.05], one per row and group."""
    return (0.01 + 0.04 * torch.rand((M, K // GROUP), generator=gen, device="cuda")).to(torch.bfloat16)


def _weights(gen, M, K, z):
    return bc.bitcos_pack_device(_trits(gen, M, K, z), _scales(gen, M, K))


def _plain_weights(gen, fmt, M, K, z):
    pack = bc.trit5_pack if fmt == "trit5" else bc.bit2_pack
    trits, scales = _trits(gen, M, K, z).cpu().numpy(), _scales(gen, M, K).view(torch.int16).cpu().numpy().view(np.uint16)
    return bc.plain_to_device(pack(trits), bc.scales_tile(scales, M, K), M, K)


def _int8_activations(gen, batch, K):
    x = torch.randint(-127, 128, (batch, K), generator=gen, device="cuda", dtype=torch.int8)
    return x, (1.0 + 3.0 * torch.rand(batch, generator=gen, device="cuda")) / 127.0


def _bf16_activations(gen, batch, K):
    """Roughly normal with a few outlier channels that carry the range, as transformer activations are."""
    x = torch.randn((batch, K), generator=gen, device="cuda")
    x[:, GROUP // 2 - 16::97] *= 24.0
    return x.to(torch.bfloat16)


def _layer_shapes(c):
    h = c["hidden"]
    return [(c["q"], h), (c["kv"], h), (c["kv"], h), (h, c["q"]), (c["ffn"], h), (c["ffn"], h), (h, c["ffn"])]


LAYER_PHASES = [0, 0, 0, 1, 2, 2, 3]
LAYER_GROUPS = [[0, 1, 2], [3], [4, 5], [6]]


def _out(batch, M):
    return torch.empty((batch, M), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    gen = _generator(seed)
    kind, z = case["kind"], case["z"]
    st = {"kind": kind}
    if kind == "gemv":
        M, K, B = case["M"], case["K"], case["batch"]
        W = _weights(gen, M, K, z) if case["fmt"] == "bitcos" else _plain_weights(gen, case["fmt"], M, K, z)
        x, xs = _int8_activations(gen, B, K)
        call = {"bitcos": bc.bitcos_gemv, "trit5": bc.trit5_gemv, "bit2": bc.bit2_gemv}[case["fmt"]]
        st.update(W=W, x=x, xs=xs, call=call, y=_out(B, M), ws=bc.make_workspace(M, K))
    elif kind == "layer":
        shapes, B = _layer_shapes(case), case["batch"]
        Ws = [_weights(gen, M, K, z) for M, K in shapes]
        wss = [bc.make_workspace(M, K) for M, K in shapes]
        st.update(act=case["act"], keep=Ws)
        # the launches that share an input: q, k and v; o; gate and up; down
        if case["act"] == "host":
            host = bc.HostPhases(list(zip(Ws, wss)), LAYER_PHASES, batch=B)
            for group in LAYER_GROUPS:
                x, xs = _int8_activations(gen, B, shapes[group[0]][1])
                for j in group:
                    host.x[j][:] = x.cpu().numpy()
                    host.x_scale[j][:B] = xs.cpu().numpy()
            st.update(host=host)
        else:
            ys, launches = [_out(B, M) for M, _ in shapes], []
            for group in LAYER_GROUPS:
                K = shapes[group[0]][1]
                x, xs = (_bf16_activations(gen, B, K), None) if case["act"] == "bf16" else _int8_activations(gen, B, K)
                launches.append(bc.MultiJobs([(Ws[j], x, xs, ys[j], wss[j]) for j in group]))
            n = len(LAYER_GROUPS)
            around = [bc.NextWeights([Ws[j] for j in group]) for group in LAYER_GROUPS]
            st.update(ys=ys, launches=launches, prev=[around[i - 1] for i in range(n)], next=[around[(i + 1) % n] for i in range(n)])
    elif kind in ("quant", "blend"):
        M, K, B = case["M"], case["K"], case["batch"]
        st.update(W=_weights(gen, M, K, z), x=_bf16_activations(gen, B, K), y=_out(B, M), ws=bc.make_workspace(M, K),
                  xq=torch.empty((B, K), dtype=torch.int8, device="cuda"),
                  xs=torch.empty((B, K // GROUP), dtype=torch.float32, device="cuda"))
    elif kind == "moe":
        E, k, h, f, T = case["experts"], case["top_k"], case["hidden"], case["ffn"], case["batch"]
        P = T * k
        experts = [bc.DeviceExperts([_weights(gen, M, K, z) for _ in range(E)]) for M, K in ((f, h), (f, h), (h, f))]
        # every token's top_k distinct experts, uniformly
        chosen = torch.rand((T, E), generator=gen, device="cuda").argsort(dim=1)[:, :k].to(torch.int32).contiguous().view(-1)
        token = torch.arange(T, dtype=torch.int32, device="cuda").repeat_interleave(k)
        x, xs = _int8_activations(gen, T, h)
        xd, xds = _int8_activations(gen, P, f)          # what the caller makes of gate and up, in list order
        st.update(experts=experts, chosen=chosen, token=token, x=x, xs=xs, xd=xd, xds=xds, E=E, T=T,
                  rows=torch.arange(P, dtype=torch.int32, device="cuda"), ys=[_out(P, M) for M in (f, f, h)],
                  ws=[bc.make_workspace(M, K, copies=min(P, E)) for M, K in ((f, h), (f, h), (h, f))])
    else:
        st.update(trits=_trits_fixed_count(gen, case["M"], case["K"], z), scales=_scales(gen, case["M"], case["K"]))
    return st


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "gemv":
        return st["call"](st["W"], st["x"], st["xs"], y=st["y"], workspace=st["ws"])[0]
    if kind == "layer":
        if st["act"] == "host":
            return st["host"].run()
        for i, jobs in enumerate(st["launches"]):
            if st["act"] == "bf16":
                bc.bitcos_gemv_multi_bf16(jobs)
            else:
                bc.bitcos_gemv_multi(jobs, prev=st["prev"][i], next=st["next"][i])
        return st["ys"]
    if kind == "quant":
        xq, xs = bc.bitcos_quantize_activations(st["x"], GROUP, xq=st["xq"], x_scale=st["xs"])
        y, _ = bc.bitcos_gemv_group_scales(st["W"], xq, xs, y=st["y"], workspace=st["ws"])
        return {"xq": xq, "x_scale": xs, "y": y}
    if kind == "blend":
        return bc.bitcos_gemv_blend_bf16(st["W"], st["x"], y=st["y"], workspace=st["ws"])
    if kind == "moe":
        ge, gb, xr, order, ng = bc.bitcos_group_pairs_device(st["chosen"], st["token"], st["E"])
        inputs = [(xr, st["x"], st["xs"]), (xr, st["x"], st["xs"]), (st["rows"], st["xd"], st["xds"])]
        for E, (rows, x, xs), y, ws in zip(st["experts"], inputs, st["ys"], st["ws"]):
            bc.bitcos_gemv_grouped_lists(E, ge, gb, ng, rows, st["T"], x, xs, y=y, workspace=ws)
        return {"order": order, "y": st["ys"]}
    W = bc.bitcos_pack_device(st["trits"], st["scales"])
    return [W.bitmap, W.signs, W.tile_off, W.scales]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _packed_bytes(fmt, M, K, z):
    Mp, G = (M + ROWS - 1) // ROWS * ROWS, K // GROUP
    if fmt == "bitcos":
        return Mp * K / 8 + (1.0 - z) * M * K / 8 + 4 * (Mp // ROWS * G + 1) + 2 * Mp * G
    if fmt == "trit5":
        return Mp * ((26 * G + 3) // 4 * 4) + 2 * Mp * G
    return Mp * K / 4 + 2 * Mp * G


def _product(fmt, M, K, B, z, x_bytes=1, x_scales=1):
    """Packed weights, activations and outputs of one product: each read or written once."""
    return {"bytes": _packed_bytes(fmt, M, K, z) + B * (x_bytes * K + 4 * x_scales + 4 * M), "flops": 2.0 * M * K * B}


def work(case):
    kind, z = case["kind"], case["z"]
    if kind == "gemv":
        parts = [_product(case["fmt"], case["M"], case["K"], case["batch"], z)]
    elif kind == "layer":
        # the launches' inputs are shared: activations counted once per launch
        x_bytes, B, shapes = (2 if case["act"] == "bf16" else 1), case["batch"], _layer_shapes(case)
        parts = [_product("bitcos", M, K, B, z, x_bytes, 0 if x_bytes == 2 else 1) for M, K in shapes]
        for group in LAYER_GROUPS:
            for j in group[1:]:
                parts[j]["bytes"] -= B * x_bytes * shapes[j][1]
    elif kind == "quant":
        M, K, B = case["M"], case["K"], case["batch"]
        parts = [_product("bitcos", M, K, B, z, 2, 0), {"bytes": B * (K + 4 * (K // GROUP)), "flops": 2.0 * B * K}]
    elif kind == "blend":
        parts = [_product("bitcos", case["M"], case["K"], case["batch"], z, 2, 0)]
    elif kind == "moe":
        E, k, h, f, T = case["experts"], case["top_k"], case["hidden"], case["ffn"], case["batch"]
        touched = E * (1.0 - (1.0 - k / E) ** T)          # experts with at least one pair, expected
        parts = []
        for M, K, rows in ((f, h, T), (f, h, T), (h, f, T * k)):
            parts.append({"bytes": touched * _packed_bytes("bitcos", M, K, z) + rows * (K + 4) + T * k * 4 * M, "flops": 2.0 * T * k * M * K})
    else:
        M, K = case["M"], case["K"]
        parts = [{"bytes": M * K + 2 * M * (K // GROUP) + _packed_bytes("bitcos", M, K, z), "flops": 0.0}]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


def tolerance(case):
    """Packed buffers and quantised codes are exact.  Products: the integer accumulators are exact, so what is left is the
    rounding of at most 200 fp32 terms per output (16-bit variant: 128 + 200 fp32 additions).  Against float64 the
    passes measure rel 2e-8 to 9e-8 and max 5e-8 to 6e-7 with a tree of sums; a running sum over 200 terms of this
    size shows about 2.5e-7 and 2.5e-6, and four times that is the limit."""
    if case["kind"] == "pack":
        return "exact"
    return {"rel": 1e-6, "max": 1e-5}
