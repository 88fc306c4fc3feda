"""Performance cases: what one denoising step of the Stable Diffusion 1.4 UNet has this library do.

Every case is one call through the public entry points: a transformer block's self- or cross-attention
(``Attention.forward``), the attention calls of a whole step side by side (``sd_attn_forward_batch``), the
feed-forward block's GEGLU (``geglu``), a group normalisation (``groupnorm``) or a 3x3 convolution
(``WinogradConv3x3``).  Sizes follow the model: an image of 8h x 8w pixels is a latent of h x w positions, halved
(rounded up) once per level of the UNet; level 0 has 320 channels in 8 heads of 40, level 1 640 (80), levels 2 and 3
1280 (160).  512 x 512 pixels (64 x 64) is the default and 768 x 768 (96 x 96) the largest; other aspect ratios give
ragged and odd token counts.  A batch of 2 is one image with guidance.
"""
import torch

from paper_2304_11267_b200 import binding as bd
from paper_2304_11267_b200 import workloads

HEADS = 8
TEXT = workloads.TEXT_TOKENS
GROUPS = 32
DTYPES = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
CODES = {"f16": bd.F16, "bf16": bd.BF16, "f32": bd.F32}
LEVEL_DIM = (40, 80, 160, 160)        # head dim at levels 0..3
LEVEL_CHANNELS = (320, 640, 1280, 1280)
# (input, output) channels of the 3x3 convolutions of each level: the residual blocks on the way down, and on the way
# up with the skip connection's channels beside the block's own
LEVEL_CONVS = (((320, 320), (640, 320), (960, 320)),
               ((320, 640), (640, 640), (960, 640), (1280, 640), (1920, 640)),
               ((640, 1280), (1280, 1280), (1920, 1280), (2560, 1280)),
               ((1280, 1280), (2560, 1280)))


def _attn(name, B, Nq, Nk, d, dtype="f16", tokens_first=False, peaked=False):
    return {"name": name, "op": "attention", "B": B, "Nq": Nq, "Nk": Nk, "d": d, "dtype": dtype,
            "tokens_first": tokens_first, "peaked": peaked}


def listed():
    return [
        # 512 x 512 with guidance, first level: most of a step's attention time
        _attn("self_4096_d40", 2, 4096, 4096, 40),
        # 768 x 768, two images with guidance, logits spread as in trained layers: the largest call
        _attn("self_9216_d40_b4", 4, 9216, 9216, 40, peaked=True),
        # the second level, where a call has fewer query tiles than the GPU has SMs
        _attn("self_1024_d80", 2, 1024, 1024, 80),
        # the innermost block: the smallest call of a step, all latency
        _attn("self_64_d160", 2, 64, 64, 160),
        # 520 x 680 pixels, second level (33 x 43), one image without guidance, bfloat16, straight from and to the
        # projections' [B, N, H * d] tensors: ragged tiles
        _attn("self_1419_d80_bf16", 1, 1419, 1419, 80, "bf16", True),
        # the first level in binary32: a reference run of the same image at full precision
        _attn("self_4096_d40_f32", 2, 4096, 4096, 40, "f32"),
        # text cross-attention at the first level: 77 keys whose last 20 are padding
        _attn("cross_4096_d40", 2, 4096, TEXT, 40),
        # text cross-attention at the third level, bfloat16 token-major
        _attn("cross_256_d160_bf16", 2, 256, TEXT, 160, "bf16", True),
        # the 32 attention calls of a step, evaluated side by side as for several requests
        {"name": "unet_step", "op": "step", "B": 2, "h": 64, "w": 64, "dtype": "f16"},
        # feed-forward block, first level: 4096 tokens, 4 x 320 hidden channels, guidance pair
        {"name": "geglu_8192_1280", "op": "geglu", "rows": 8192, "C": 1280, "dtype": "f16"},
        # the residual blocks' normalisation, first level
        {"name": "groupnorm_320_64x64", "op": "groupnorm", "N": 2, "C": 320, "h": 64, "w": 64, "dtype": "f16"},
        # the residual blocks' convolution, first level
        {"name": "conv_320_64x64", "op": "conv", "N": 2, "h": 64, "w": 64, "C": 320, "K": 320},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def _latent(rng, most=96):
    """An image's latent: any size of 32 positions a side and more, up to `most` x `most`."""
    return _log_int(rng, 32, most), _log_int(rng, 32, most)


def _level(rng, h, w):
    lv = rng.choice((0, 0, 1, 1, 2, 3))
    for _ in range(lv):
        h, w = (h + 1) // 2, (w + 1) // 2
    return lv, h, w


def draw(rng):
    op = rng.choices(("self", "cross", "step", "geglu", "groupnorm", "conv"), (30, 20, 8, 12, 15, 15))[0]
    if op == "step":   # (a step costs a dozen times its largest call: smaller images and batches)
        h, w = _latent(rng, 64)
        return {"op": "step", "B": rng.choice((1, 2)), "h": h, "w": w, "dtype": rng.choice(("f16", "bf16"))}
    h, w = _latent(rng)
    lv, h, w = _level(rng, h, w)
    B = rng.choice((1, 2, 2, 3, 4))
    if op in ("self", "cross"):
        dtype = rng.choices(("f16", "bf16", "f32"), (6, 3, 1))[0]
        if dtype == "f32":   # (no dearer than the listed binary32 call)
            B = min(B, 2)
            h, w = min(h, 64), min(w, 64)
        # long prompts are encoded as two or three pieces of 77 tokens
        Nk = h * w if op == "self" else rng.choice((TEXT, TEXT, TEXT, 2 * TEXT, 3 * TEXT))
        c = _attn("", B, h * w, Nk, LEVEL_DIM[lv], dtype, rng.random() < 0.4, rng.random() < 0.3)
    elif op == "geglu":
        c = {"op": op, "rows": B * h * w, "C": 4 * LEVEL_CHANNELS[lv], "dtype": rng.choice(("f16", "f16", "f32"))}
    elif op == "groupnorm":
        ch = LEVEL_CHANNELS[lv] * (1 if rng.random() < 0.7 else 2)
        c = {"op": op, "N": B, "C": ch, "h": h, "w": w, "dtype": rng.choice(("f16", "f16", "f32"))}
    else:
        C, K = rng.choice(LEVEL_CONVS[lv])
        c = {"op": op, "N": B, "h": h, "w": w, "C": C, "K": K}
    c.pop("name", None)
    return c


def _step_calls(c):
    """(Nq, Nk, d) of the attention calls of a step: every block has one self- and one cross-attention."""
    calls, h, w = [], c["h"], c["w"]
    for _, d, blocks in workloads.UNET_BLOCKS:
        calls += [(h * w, h * w, d), (h * w, TEXT, d)] * blocks
        h, w = (h + 1) // 2, (w + 1) // 2
    return calls


def _qkv(gen, B, Nq, Nk, d, dtype, tokens_first=False, peaked=False):
    def normal(n, mult=1.0):
        t = torch.randn(B, HEADS, n, d, generator=gen, device="cuda") * mult
        if n == TEXT and Nq != Nk:   # text padded to 77 tokens: the padding rows are alike
            t[:, :, -workloads.PADDING_ROWS:] = t[:, :, -workloads.PADDING_ROWS:-workloads.PADDING_ROWS + 1].clone()
        return (t.transpose(1, 2) if tokens_first else t).to(dtype).contiguous()
    return normal(Nq, 4.0 if peaked else 1.0), normal(Nk), normal(Nk)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op = case["op"]
    s = {"op": op}
    if op == "attention":
        s["attn"] = bd.Attention(layout=bd.LAYOUT_BNHD if case["tokens_first"] else bd.LAYOUT_BHND)
        s["qkv"] = _qkv(gen, case["B"], case["Nq"], case["Nk"], case["d"], DTYPES[case["dtype"]], case["tokens_first"],
                        case["peaked"])
    elif op == "step":
        s["attn"] = bd.Attention()
        s["tensors"] = [_qkv(gen, case["B"], Nq, Nk, d, DTYPES[case["dtype"]]) for Nq, Nk, d in _step_calls(case)]
        s["outs"] = [torch.empty_like(q) for q, _, _ in s["tensors"]]
        s["problems"] = bd.make_problems(
            [(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), case["B"], HEADS, q.shape[2], k.shape[2], q.shape[3],
              q.shape[3] ** -0.5) for (q, k, v), o in zip(s["tensors"], s["outs"])])
        s["dtype"] = CODES[case["dtype"]]
    elif op == "geglu":
        s["x"] = torch.randn(case["rows"], 2 * case["C"], generator=gen, device="cuda").to(DTYPES[case["dtype"]])
    elif op == "groupnorm":
        dtype = DTYPES[case["dtype"]]
        n = case["C"]
        s["x"] = (torch.randn(case["N"], n, case["h"], case["w"], generator=gen, device="cuda") * 1.7 + 0.4).to(dtype)
        s["gamma"] = (1.0 + 0.3 * torch.randn(n, generator=gen, device="cuda")).to(dtype)
        s["beta"] = (0.2 * torch.randn(n, generator=gen, device="cuda")).to(dtype)
    else:
        N, h, w, C, K = (case[k] for k in ("N", "h", "w", "C", "K"))
        s["x"] = torch.randn(N, h, w, C, generator=gen, device="cuda").half()
        weight = (torch.randn(K, 3, 3, C, generator=gen, device="cuda") / (9.0 * C) ** 0.5).half()
        bias = (0.1 * torch.randn(K, generator=gen, device="cuda")).half()
        s["layer"] = bd.WinogradConv3x3(weight, bias)
    return s


def run(s):
    op = s["op"]
    if op == "attention":
        return s["attn"].forward(*s["qkv"])
    if op == "step":
        rc = bd.sd_attn_forward_batch(s["attn"].handle, s["problems"], s["dtype"], torch.cuda.current_stream().cuda_stream)
        if rc != bd.OK:
            raise bd.SdAttnError(rc, "sd_attn_forward_batch")
        return s["outs"]
    if op == "geglu":
        return bd.geglu(s["x"])
    if op == "groupnorm":
        return bd.groupnorm(s["x"], GROUPS, 1e-5, s["gamma"], s["beta"])
    return s["layer"](s["x"])


def work(case):
    es = 4 if case.get("dtype") == "f32" else 2
    op = case["op"]
    if op in ("attention", "step"):
        calls = _step_calls(case) if op == "step" else [(case["Nq"], case["Nk"], case["d"])]
        bh = case["B"] * HEADS
        return {"bytes": sum(2 * es * bh * d * (Nq + Nk) for Nq, Nk, d in calls),
                "flops": sum(4 * bh * d * Nq * Nk for Nq, Nk, d in calls)}
    if op == "geglu":   # the gate's error function is about thirty operations
        n = case["rows"] * case["C"]
        return {"bytes": 3 * es * n, "flops": 30 * n}
    if op == "groupnorm":
        n = case["N"] * case["C"] * case["h"] * case["w"]
        return {"bytes": 2 * es * n + 2 * es * case["C"], "flops": 7 * n}
    # a 3x3 convolution in the domain of F(4x4, 3x3): 36 products per channel pair for 16 outputs
    N, h, w, C, K = (case[k] for k in ("N", "h", "w", "C", "K"))
    tiles = N * ((h + 3) // 4) * ((w + 3) // 4)
    return {"bytes": 2 * (N * h * w * (C + K) + 9 * C * K + K), "flops": 2 * 36 * tiles * C * K}


def tolerance(case):
    op, dtype = case["op"], case.get("dtype")
    if op in ("attention", "step"):   # weights and result are each rounded once to the storage type
        return {"rel": {"f16": 1e-3, "bf16": 6e-3, "f32": 1e-5}[dtype]}
    if op == "conv":   # the transforms amplify the binary16 rounding of the transformed values: 3e-3 of the result's r.m.s.
        return {"rel": 6e-3, "max": 0.1}
    return {"rel": 5e-4 if dtype == "f16" else 1e-5}   # binary32 arithmetic, rounded once
