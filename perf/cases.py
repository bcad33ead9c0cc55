"""The work that users of this library have it do, as measurable cases through the public binding (``paper_2609_28358_b200.mq``).

A case is one convolution layer and one job on it:

  train    a training step of the layer from full-precision tensors: X, W and G_Y quantized once each, then Y, G_X and G_W
  replay   the same step when the activation exists only in its stored form (latent replay): W and G_Y quantized, then Y, G_X, G_W
  chain    a layer inside a chain of quantized layers: the forward result leaves as the next layer's stored activation, the input
           gradient as the previous layer's stored gradient, and the weight gradient is taken from the stored tensors
  forward  inference with stored weights: X quantized, then Y
  encode   X quantized and expanded by the channel-batch-first im2col

Formats are named by their element type ("e2m1"), "ts16" being the paper's own format (E2M1 elements, E4M3 scale per 16 x 16
block, fp32 tensor scale).  Tensors are drawn on the GPU from the seed, with the distributions of ``inputs.py``.
"""
import math

import torch

from paper_2609_28358_b200 import mq

_FMT = {"e4m3": mq.E4M3, "e5m2": mq.E5M2, "e2m1": mq.E2M1, "e3m2": mq.E3M2, "e2m3": mq.E2M3, "e3m2_p6": mq.E3M2_P6, "e2m3_p6": mq.E2M3_P6,
        "ts16": mq.E2M1}
_BITS = {"e4m3": 8, "e5m2": 8, "e2m1": 4, "e3m2": 8, "e2m3": 8, "e3m2_p6": 6, "e2m3_p6": 6, "ts16": 4}
_BLOCK = {"tile32": mq.TILE32, "line32": mq.LINE32}
_ACT = {"none": mq.ACT_NONE, "relu": mq.ACT_RELU, "silu": mq.ACT_SILU}


def _case(job, n, cin, hw, cout, k, stride, x_fmt, w_fmt=None, dy_fmt=None, values="relu", layout="nchw", block="tile32", stochastic=False, act="relu"):
    return {"job": job, "n": n, "cin": cin, "h": hw, "w": hw, "cout": cout, "k": k, "stride": stride, "x_fmt": x_fmt, "w_fmt": w_fmt or x_fmt,
            "dy_fmt": dy_fmt or x_fmt, "values": values, "layout": layout, "block": block, "stochastic": stochastic, "act": act}


def listed():
    return [
        # a single small convolution, as in fine-tuning at the edge: launches and host work are what it costs
        dict(_case("train", 8, 32, 32, 64, 3, 1, "e4m3", "e4m3", "e5m2"), name="train_edge_c32_hw32"),
        # first down-sampling layer of a nano-width detector backbone (batch 16, 640 x 640 images): few channels, large image
        dict(_case("train", 16, 16, 320, 32, 3, 2, "e4m3", "e4m3", "e5m2", values="silu"), name="train_detector_down_c16_hw320"),
        # 4-bit training of a mid-size layer whose activations have outliers
        dict(_case("train", 32, 64, 80, 128, 3, 1, "e2m1", values="outliers"), name="train_e2m1_outliers_c64_hw80"),
        # latent replay: a late layer trained on activations kept only in 4 bits
        dict(_case("replay", 256, 512, 14, 512, 3, 1, "e2m1"), name="replay_e2m1_c512_hw14"),
        # the largest layer of the throughput sweep
        dict(_case("train", 256, 512, 56, 512, 3, 1, "e4m3", values="gauss"), name="train_e4m3_c512_hw56"),
        # a down-sampling layer of a wide network in 4 bits
        dict(_case("train", 256, 256, 28, 256, 3, 2, "e2m1", values="gauss"), name="train_e2m1_stride2_c256_hw28"),
        # a pointwise layer: as many bytes as a 3 x 3 one, a ninth of its arithmetic
        dict(_case("train", 256, 256, 56, 256, 1, 1, "e4m3", values="gauss"), name="train_pointwise_c256_hw56"),
        # the paper's own format with its stochastically rounded gradient and the tensor maxima of the previous step
        dict(_case("train", 256, 256, 28, 256, 3, 1, "ts16", stochastic=True), name="train_paper_format_c256_hw28"),
        # 6-bit activations in packed storage with 8-bit weights and gradients, tensors kept channel-fastest
        dict(_case("train", 256, 256, 28, 256, 3, 1, "e3m2_p6", "e4m3", "e5m2", layout="hwnc"), name="train_e3m2_packed_c256_hw28"),
        # a layer inside a chain of quantized layers
        dict(_case("chain", 256, 256, 28, 256, 3, 1, "e4m3", "e4m3", "e5m2"), name="chain_e4m3_c256_hw28"),
        # sizes that no tile divides: the last batch of an epoch, a 96-channel layer, an odd image
        dict(_case("train", 50, 96, 27, 160, 3, 1, "e2m1"), name="train_e2m1_ragged_c96_hw27"),
        # quantizer and explicit im2col, for a user whose own GEMM follows
        dict(_case("encode", 256, 128, 56, 128, 3, 1, "e4m3"), name="encode_e4m3_c128_hw56"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Mostly multiples of 16 or 32, as networks have them; now and then any number."""
    c = _log_int(rng, lo, hi)
    step = rng.choice((1, 16, 32, 32, 32, 64))
    return max(lo, min(hi, (c + step // 2) // step * step))


def draw(rng):
    top = max((work(c) for c in listed()), key=lambda v: v["flops"])
    while True:
        job = rng.choice(("train", "train", "train", "train", "replay", "chain", "chain", "forward", "encode"))
        fmts = [("e4m3", "e4m3", "e4m3"), ("e4m3", "e4m3", "e5m2"), ("e2m1", "e2m1", "e2m1"), ("e2m1", "e2m1", "e2m1")]
        if job in ("train", "replay", "chain"):
            fmts.append(("ts16", "ts16", "ts16"))
        if job in ("train", "encode", "forward"):
            fmts.append(rng.choice((("e3m2_p6", "e4m3", "e5m2"), ("e2m3", "e2m3", "e2m3"))))
        x, w, dy = rng.choice(fmts)
        k = rng.choice((1, 3, 3, 3, 5))
        case = _case(job, _log_int(rng, 8, 256), _channels(rng, 16, 512), _log_int(rng, 7, 160), _channels(rng, 16, 512), k, rng.choice((1, 1, 2)), x, w, dy,
                     values=rng.choice(("relu", "silu", "gauss", "outliers")), layout=rng.choice(("nchw", "nchw", "nchw", "hwnc")),
                     block="line32" if job == "forward" and rng.random() < 0.5 else "tile32", stochastic=job in ("train", "replay") and rng.random() < 0.25,
                     act=rng.choice(("relu", "silu", "none")))
        if rng.random() < 0.3:
            case["w"] = max(7, case["h"] * rng.choice((3, 5, 7)) // 4)
        if case["h"] < k or case["w"] < k:
            continue
        need = work(case)
        # a 4-bit layer with a channel count that is no multiple of 64 is a small one
        most = top["flops"] / (4 if min(_BITS[x], _BITS[w], _BITS[dy]) > 4 or (case["cin"] % 64 == 0 and case["cout"] % 64 == 0) else 400)
        if need["bytes"] <= top["bytes"] / 2 and need["flops"] <= most:
            return case


def _desc(c):
    return mq.ConvDesc(c["n"], c["cin"], c["h"], c["w"], c["cout"], c["k"], c["k"], c["stride"], c["stride"], c["k"] // 2, c["k"] // 2)


def _out_hw(c):
    return tuple((v + 2 * (c["k"] // 2) - c["k"]) // c["stride"] + 1 for v in (c["h"], c["w"]))


def _x(shape, values, gen):
    z = torch.randn(shape, generator=gen, device="cuda")
    if values == "gauss":
        return z
    if values == "silu":
        return torch.nn.functional.silu(z)
    z.clamp_(min=0.0)
    if values == "outliers":  # one element in a hundred is fifty times as large
        z[torch.rand(shape, generator=gen, device="cuda") < 0.01] *= 50.0
    return z


def _quantize(c, desc, role, src, fmt, amax=None, seed=None):
    layout = mq.HWNC if c["layout"] == "hwnc" else mq.NCHW
    if fmt == "ts16":
        return mq.quantize_ts(desc, role, src, src_layout=layout, amax_in=amax, seed=seed)
    if seed is not None:
        return mq.quantize_sr(desc, role, _FMT[fmt], src, seed, src_layout=layout)
    return mq.quantize(desc, role, _FMT[fmt], src, src_layout=layout, block=_BLOCK[c["block"]])


def prepare(case, seed):
    c, desc = case, _desc(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    ho, wo = _out_hw(c)
    n, ci, co, k = c["n"], c["cin"], c["cout"], c["k"]
    hwnc = c["layout"] == "hwnc"
    st = {"case": c, "desc": desc, "seed": int(seed)}
    x = _x((c["h"], c["w"], n, ci) if hwnc else (n, ci, c["h"], c["w"]), c["values"], gen)
    w = torch.randn((co, k, k, ci) if hwnc else (co, ci, k, k), generator=gen, device="cuda") * math.sqrt(2.0 / (ci * k * k))
    sigma = 1.0 if c["values"] == "gauss" else 1e-3
    dy = torch.randn((ho, wo, n, co) if hwnc else (n, co, ho, wo), generator=gen, device="cuda") * sigma if c["job"] in ("train", "replay", "chain") else None
    job = c["job"]
    if job in ("train", "forward", "encode"):
        st["x"] = x
    if job in ("train", "replay"):
        st["w"], st["dy"] = w, dy
    if c["x_fmt"] == "ts16":  # the previous step's maxima, a little off this step's
        st["x_amax"], st["dy_amax"] = x.abs().max().reshape(1) * 0.98, dy.abs().max().reshape(1) * 1.02
    if job in ("replay", "chain"):
        st["xq"] = _quantize(c, desc, mq.ROLE_X, x, c["x_fmt"])
    if job in ("chain", "forward"):
        st["wq"] = _quantize(c, desc, mq.ROLE_W, w, c["w_fmt"])
    if job == "chain":
        st["dyq"] = _quantize(c, desc, mq.ROLE_DY, dy, c["dy_fmt"])
        # maxima of the previous step's emitted tensors: a convolution of the operands' spread
        gain = math.sqrt(ci * k * k) * float(x.square().mean().sqrt()) * math.sqrt(2.0 / (ci * k * k))
        st["y_amax"] = torch.full((1,), 5.0 * gain, device="cuda")
        st["dx_amax"] = torch.full((1,), 5.0 * sigma * math.sqrt(2.0 * co / (ci * c["stride"] ** 2)), device="cuda")
    return st


def _stored(name, q):
    out = {name + "_codes": q.codes, name + "_scales": q.scales}
    if q.tensor_scale is not None:
        out[name + "_tensor_scale"] = q.tensor_scale
    return out


def run(state):
    c, desc = state["case"], state["desc"]
    layout = mq.HWNC if c["layout"] == "hwnc" else mq.NCHW
    job, out = c["job"], {}
    xq, wq, dyq = state.get("xq"), state.get("wq"), state.get("dyq")
    if xq is None:
        xq = _quantize(c, desc, mq.ROLE_X, state["x"], c["x_fmt"], amax=state.get("x_amax"))
        out.update(_stored("x", xq))
    if job == "encode":
        out["cols_codes"], out["cols_scales"] = mq.cbf_im2col(desc, xq)
        return out
    if wq is None:
        wq = _quantize(c, desc, mq.ROLE_W, state["w"], c["w_fmt"])
        out.update(_stored("w", wq))
    if job == "forward":
        out["y"] = mq.conv_fwd(desc, xq, wq, layout=layout)
        return out
    if dyq is None:
        dyq = _quantize(c, desc, mq.ROLE_DY, state["dy"], c["dy_fmt"], amax=state.get("dy_amax"), seed=state["seed"] if c["stochastic"] else None)
        out.update(_stored("dy", dyq))
    if job == "chain":
        if c["x_fmt"] == "ts16":
            out.update(_stored("y", mq.conv_fwd_ts(desc, xq, wq, state["y_amax"], act=_ACT[c["act"]])))
            out.update(_stored("dx", mq.conv_bwd_data_ts(desc, wq, dyq, state["dx_amax"])))
        else:
            out.update(_stored("y", mq.conv_fwd_mx(desc, xq, wq, _FMT[c["x_fmt"]], act=_ACT[c["act"]])))
            out.update(_stored("dx", mq.conv_bwd_data_mx(desc, wq, dyq, _FMT[c["dy_fmt"]])))
    else:
        out["y"] = mq.conv_fwd(desc, xq, wq, layout=layout)
        out["dx"] = mq.conv_bwd_data(desc, wq, dyq, layout=layout)
    out["dw"] = mq.conv_bwd_weight(desc, xq, dyq, layout=layout)
    return out


def work(case):
    c = case
    ho, wo = _out_hw(c)
    job = c["job"]
    n_x, n_w, n_y = c["n"] * c["cin"] * c["h"] * c["w"], c["cout"] * c["cin"] * c["k"] ** 2, c["n"] * c["cout"] * ho * wo
    gemm = 2.0 * n_y * c["cin"] * c["k"] ** 2

    def st(n, fmt):
        return n * _BITS[fmt] / 8.0

    x, w, dy = st(n_x, c["x_fmt"]), st(n_w, c["w_fmt"]), st(n_y, c["dy_fmt"])
    if job == "encode":
        return {"bytes": 4.0 * n_x + x + st(n_y // c["cout"] * c["cin"] * c["k"] ** 2, c["x_fmt"]), "flops": 0.0}
    if job == "forward":
        return {"bytes": 4.0 * n_x + x + w + 4.0 * n_y, "flops": gemm}
    if job == "chain":
        return {"bytes": x + w + dy + st(n_y, c["x_fmt"]) + st(n_x, c["dy_fmt"]) + 4.0 * n_w, "flops": 3 * gemm}
    first = x if job == "replay" else 4.0 * n_x + x
    return {"bytes": first + 4.0 * n_w + w + 4.0 * n_y + dy + 4.0 * n_y + 4.0 * n_x + 4.0 * n_w, "flops": 3 * gemm}


def tolerance(case):
    # Codes, scales and im2col bytes are exact.  fp32 results are sums of up to 800 thousand products: against 64-bit sums, and with
    # channels or samples in another order, they differ by up to 8e-7 (2-norm) and 4.2e-6 (largest).
    if case["job"] == "encode":
        return "exact"
    tol = {"rel": 4e-6, "max": 2e-5}
    if case["job"] == "chain":
        tol["differ"] = 1e-4  # a sum that moves by its rounding moves a few codes to their neighbours (one in a million seen)
    return tol
