"""Calls that programs make of this framework, for timing and comparing.

Every case is a call (or the few calls of one step) through the public Python
entry points of paper_2608_01653_gb300 on seeded inputs. The kinds:

  f16_layer   one DH 1x1 layer from FP16 activations to float32 (hatq.layer):
              a layer used by itself inside a float model
  i8_layer    one convolution on INT8 activations with its input transform
              (hatq.layer), any activation of the library
  analysis    the encoder's image-to-latent chain (Chain.forward)
  entropy     the hyperprior chain and the eight context-slice chains of the
              entropy model (Chain.forward, one chain after another)
  quantize    the activation transform and quantization pass by itself
              (hatq.quantize_act), as calibration and mixed-precision models use it
  gdn_layer   an encoder layer emitting the preactivation, then the GDN / IGDN
              transition (hatq.conv2d_i8, hatq.gdn)
  synthesis   the decoder direction: latents through three transposed
              convolutions (hatq.quantize_act, hatq.conv_transpose2d_i8)
  subpixel    a decoder layer with the sub-pixel rearrangement
              (hatq.conv2d_i8_subpixel)
  affine      post-training quantization with dynamic affine activations
              (hatq.quantize_act_affine, hatq.conv2d_affine)

A program loads its model once and calls it on many images, so the weights of
a kind are the same for every seed and kept between preparations; all
activations are drawn from the seed. Output and scratch buffers are allocated
once per state, as Chain.alloc does for its users.
"""
from __future__ import annotations

import functools
import math
from dataclasses import dataclass

import numpy as np
import torch

from paper_2608_01653_gb300 import hatq
from paper_2608_01653_gb300.chain import Chain

DEV = "cuda"
S_IMAGE = 1.0 / 127.0     # scale of image codes (pixels in [0, 1])
S_LATENT = 0.1            # scale of latent codes
S_ACT = 0.05              # scale of INT8 activations
W_STD = 0.0363            # standard deviation of the drawn weights (Laplace 0.02 times a log-normal gain)
RANGE = 10.0              # a scale maps this many standard deviations to code 127


def listed():
    return [
        # one 1x1 layer on a 16x16 feature map: the smallest call, latency alone
        dict(name="f16_layer_16x16", kind="f16_layer", n=1, h=16, w=16, c=128),
        # one strided layer on a feature map of a small picture
        dict(name="i8_layer_256", kind="i8_layer", n=1, h=256, w=256, c=192, c_out=192, k=5, stride=2, act="none"),
        # encoding one picture of a usual test set
        dict(name="analysis_512x768", kind="analysis", n=1, h=512, w=768),
        # encoding one picture of odd size, unpadded
        dict(name="analysis_1361x2041", kind="analysis", n=1, h=1361, w=2041),
        # encoding a batch of 4K pictures: the largest call
        dict(name="analysis_4k_b8", kind="analysis", n=8, h=2160, w=3840),
        # the entropy model of one small picture: many short launches
        dict(name="entropy_32x48", kind="entropy", n=1, h=32, w=48),
        # the entropy model of a batch of 4K pictures
        dict(name="entropy_4k_b8", kind="entropy", n=8, h=135, w=240),
        # the transform pass over a large INT8 feature map
        dict(name="quantize_i8_1080p_b8", kind="quantize", dtype="i8", dynamic=False, n=8, h=1080, w=1920, c=192, hb=64),
        # an encoder layer with GDN on a batch of 1080p feature maps
        dict(name="gdn_layer_1080p_b4", kind="gdn_layer", n=4, h=1080, w=1920, inverse=False),
        # decoding one 1080p picture
        dict(name="synthesis_1080p", kind="synthesis", n=1, h=68, w=120),
        # a sub-pixel decoder layer on a batch
        dict(name="subpixel_270x480_b8", kind="subpixel", n=8, h=270, w=480),
        # a post-training-quantized layer with an odd feature map
        dict(name="affine_541x961", kind="affine", n=1, h=541, w=961),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["f16_layer", "i8_layer", "analysis", "analysis", "entropy", "entropy", "quantize", "gdn_layer",
                       "synthesis", "subpixel", "affine"])
    case = dict(kind=kind, n=size(1, 8))
    if kind == "f16_layer":
        case.update(h=size(3, 135), w=size(3, 240), c=rng.choice([64, 128, 192, 320]))
    elif kind == "i8_layer":
        c = rng.choice([32, 64, 128, 192, 224, 320])
        act = rng.choice(["none", "relu"] if c == 128 else ["none", "relu", "silu", "gelu"])
        case.update(h=size(9, 540), w=size(9, 960), c=c, c_out=rng.choice([64, 192, 320]), k=rng.choice([1, 3, 5]),
                    stride=rng.choice([1, 2]), act=act)
    elif kind == "analysis":
        case.update(h=size(64, 2160), w=size(64, 3840))
    elif kind == "entropy":
        case.update(h=size(5, 135), w=size(5, 240))
    elif kind == "quantize":
        c, hb = rng.choice([(192, 64), (320, 64), (128, 128), (640, 128), (224, 32), (256, 256)])
        case.update(dtype=rng.choice(["i8", "f16"]), dynamic=rng.choice([False, True]), h=size(16, 1080), w=size(16, 960),
                    c=c, hb=hb)
    elif kind == "gdn_layer":
        case.update(h=size(17, 1080), w=size(17, 1920), inverse=rng.choice([False, True]))
    elif kind == "synthesis":
        case.update(h=size(4, 135), w=size(4, 240))
    elif kind == "subpixel":
        case.update(h=size(5, 270), w=size(5, 480))
    else:
        case.update(h=size(17, 541), w=size(17, 961))
    return case


# ------------------------------------------------------------------ models

def block(c):
    """Hadamard block along c channels: the largest power of two dividing c, at most 128."""
    return min(128, c & -c)


@dataclass(frozen=True)
class Layer:
    c_in: int
    c_out: int
    k: int
    stride: int
    pad: int
    form: str
    act: str
    hb_in: int
    hb_out: int

    def out_hw(self, h, w):
        return (h + 2 * self.pad - self.k) // self.stride + 1, (w + 2 * self.pad - self.k) // self.stride + 1

    def macs(self, n, h, w):
        ho, wo = self.out_hw(h, w)
        return n * ho * wo * self.c_out * self.c_in * self.k * self.k

    def weight_bytes(self):
        return self.c_out * self.c_in * self.k * self.k


def layer(c_in, c_out, k, stride, form, act):
    return Layer(c_in, c_out, k, stride, k // 2, form, act, block(c_in) if form == "DH" else 0,
                 block(c_out) if form == "WH" else 0)


ANALYSIS = (layer(3, 192, 5, 2, "WH", "relu"), layer(192, 192, 5, 2, "DH", "relu"), layer(192, 192, 5, 2, "DH", "relu"),
            layer(192, 320, 5, 2, "DH", "none"))


@functools.lru_cache(None)
def entropy_layers():
    """The hyperprior chain and eight context-slice chains; a seeded 30 % of the layers are WH."""
    mask = np.random.Generator(np.random.PCG64(3)).random(27) < 0.3
    forms = iter(["WH" if m else "DH" for m in mask])
    chains = [tuple(layer(ci, co, k, 1, next(forms), act)
                    for ci, co, k, act in ((320, 640, 3, "relu"), (640, 640, 3, "relu"), (640, 640, 1, "none")))]
    for _ in range(8):
        chains.append(tuple(layer(ci, co, 3, 1, next(forms), act)
                            for ci, co, act in ((32, 224, "relu"), (224, 128, "relu"), (128, 32, "none"))))
    return tuple(chains)


def weights(c_out, k, c_in, seed):
    """(OHWI float32 weights, bias): Laplace with a log-normal gain per output channel."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lam = rng.lognormal(0.0, 0.5, size=c_out)
    w = rng.laplace(0.0, 0.02, size=(c_out, k, k, c_in)) * lam[:, None, None, None]
    return w.astype(np.float32), rng.laplace(0.0, 0.01, size=c_out).astype(np.float32)


def scale(std):
    return float(np.float32(RANGE * std / 127.0))


def out_std(fan_in, std):
    return W_STD * math.sqrt(fan_in) * std


def make_chain(layers, seed, s_in, std):
    """A Chain whose scales follow the activations' standard deviation through the layers."""
    params, scales, plan = [], [], []
    s_x = s_in if layers[0].form == "WH" else scale(std)
    for i, L in enumerate(layers):
        params.append(weights(L.c_out, L.k, L.c_in, seed + i))
        std = out_std(L.c_in * L.k * L.k, std) * (0.7 if L.act == "relu" else 1.0)
        scales.append(dict(s_x=s_x, s_out=scale(std)))
        s_x = scale(std)
        plan.append(layers[i + 1].hb_in if i + 1 < len(layers) and layers[i + 1].form == "DH" else 0)
    return Chain(layers, params, scales, plan)


@functools.lru_cache(None)
def analysis_chain():
    return make_chain(ANALYSIS, 100, S_IMAGE, 0.57)


@functools.lru_cache(None)
def entropy_model():
    return tuple(make_chain(c, 200 + 10 * i, S_LATENT, 3.0) for i, c in enumerate(entropy_layers()))


@functools.lru_cache(None)
def f16_model(c):
    w, b = weights(c, 1, c, 300)
    return hatq.prepare_weights(hatq.make_desc(c, c, 1, 1, 0, "DH", hb_in=block(c)), w, b, F16_S_X, 1.0, "none", 0, True)


F16_S_X = float(np.float32(0.35))     # operand scale of the FP16-entry layers


def i8_layer(case):
    return layer(case["c"], case["c_out"], case["k"], case["stride"], "DH", case["act"])


@functools.lru_cache(None)
def i8_model(L):
    w, b = weights(L.c_out, L.k, L.c_in, 400)
    s = scale(out_std(L.c_in * L.k * L.k, 1.5))
    hb_next = min(64, block(L.c_out))
    desc = hatq.make_desc(L.c_in, L.c_out, L.k, L.stride, L.pad, "DH", hb_in=L.hb_in)
    if L.act in ("silu", "gelu"):
        return hatq.prepare_weights(desc, w, b, scale(1.5), s, L.act, hb_next, s_z=s, s_u=s)
    return hatq.prepare_weights(desc, w, b, scale(1.5), s, L.act, hb_next)


GDN_C, GDN_S_Z, GDN_S_U = 192, float(np.float32(0.05)), float(np.float32(0.04))


@functools.lru_cache(None)
def gdn_model(inverse):
    """A 5x5 stride-2 layer emitting preactivation codes, and GDN parameters in the usual range."""
    w, b = weights(GDN_C, 5, GDN_C, 500)
    L = hatq.prepare_weights(hatq.make_desc(GDN_C, GDN_C, 5, 2, 2, "DH", hb_in=64), w, b, scale(0.5), GDN_S_Z, "none", 0)
    rng = np.random.Generator(np.random.PCG64(501))
    beta, gamma = 0.5 + rng.random(GDN_C), 0.01 * np.abs(rng.standard_normal((GDN_C, GDN_C)))
    g = hatq.prepare_gdn(GDN_C, beta, gamma, GDN_S_Z, GDN_S_U * (4.0 if inverse else 1.0), inverse, 0.05, 64)
    return L, g


SYNTHESIS = ((320, 192, "relu"), (192, 192, "relu"), (192, 192, "none"))    # 5x5 stride 2, output padding 1


@functools.lru_cache(None)
def synthesis_model():
    std, s_x, out = 3.0, scale(3.0), []
    for i, (ci, co, act) in enumerate(SYNTHESIS):
        w, b = weights(co, 5, ci, 600 + i)
        std = out_std(ci * 25 / 4, std) * (0.7 if act == "relu" else 1.0)
        desc = hatq.make_desc(ci, co, 5, 2, 2, "DH", hb_in=64)
        out.append(hatq.prepare_weights_transposed(desc, 1, w, b, s_x, scale(std), act, 64 if i < 2 else 0))
        s_x = scale(std)
    return tuple(out)


SUBPIXEL = layer(192, 768, 3, 1, "DH", "relu")


@functools.lru_cache(None)
def subpixel_model():
    w, b = weights(SUBPIXEL.c_out, 3, SUBPIXEL.c_in, 700)
    return hatq.prepare_weights(hatq.desc_from_spec(SUBPIXEL), w, b, scale(0.5),
                                scale(out_std(SUBPIXEL.c_in * 9, 0.5)), "relu", 0)


AFFINE = layer(192, 192, 5, 2, "DH", "relu")


@functools.lru_cache(None)
def affine_model():
    w, b = weights(AFFINE.c_out, 5, AFFINE.c_in, 800)
    return hatq.prepare_weights_affine(hatq.desc_from_spec(AFFINE), w, b, "relu")


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def image_codes(g, n, h, w):
    """Pixels uniform in [0, 1] as codes rint(127 x)."""
    return torch.randint(0, 128, (n, h, w, 3), generator=g, device=DEV, dtype=torch.int8)


def activations(g, n, h, w, c, std=1.0):
    """Yields one picture at a time: Gaussian with a log-normal scale per channel, heavy-tailed through it."""
    s = torch.exp(0.5 * torch.randn(c, generator=g, device=DEV)) * std
    for _ in range(n):
        yield torch.randn((h, w, c), generator=g, device=DEV) * s


def codes(g, n, h, w, c, std, s):
    x = torch.empty((n, h, w, c), dtype=torch.int8, device=DEV)
    for i, a in enumerate(activations(g, n, h, w, c, std)):
        x[i] = torch.clamp(torch.round(a / s), -127, 127).to(torch.int8)
    return x


def halves(g, n, h, w, c, std):
    x = torch.empty((n, h, w, c), dtype=torch.float16, device=DEV)
    for i, a in enumerate(activations(g, n, h, w, c, std)):
        x[i] = a.to(torch.float16)
    return x


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    n, h, w = case["n"], case["h"], case["w"]

    def i8(*shape):
        return torch.empty(shape, dtype=torch.int8, device=DEV)

    st = dict(case=case)
    if kind == "f16_layer":
        c = case["c"]
        st.update(P=f16_model(c), x=halves(g, n, h, w, c, 1.0), scratch=i8(n * h * w * c),
                  y=torch.empty((n, h, w, c), dtype=torch.float32, device=DEV))
    elif kind == "i8_layer":
        P = i8_model(i8_layer(case))
        st.update(P=P, x=codes(g, n, h, w, case["c"], 1.5, S_ACT), scratch=i8(n * h * w * case["c"]),
                  y=i8(*P.out_shape(n, h, w)))
    elif kind == "analysis":
        ch = analysis_chain()
        outs, scratch = ch.alloc(n, h, w, DEV)
        st.update(chain=ch, x=image_codes(g, n, h, w), outs=outs, scratch=scratch)
    elif kind == "entropy":
        st.update(runs=[])
        for ch in entropy_model():
            outs, scratch = ch.alloc(n, h, w, DEV)
            st["runs"].append((ch, codes(g, n, h, w, ch.layers[0].c_in, 3.0, S_LATENT), outs, scratch))
    elif kind == "quantize":
        c = case["c"]
        x = codes(g, n, h, w, c, 1.5, S_ACT) if case["dtype"] == "i8" else halves(g, n, h, w, c, 1.5)
        st.update(x=x, y=i8(n, h, w, c), s_used=torch.empty(1, dtype=torch.float32, device=DEV),
                  workspace=torch.empty(64, dtype=torch.uint8, device=DEV))
    elif kind == "gdn_layer":
        L, gd = gdn_model(case["inverse"])
        shape = L.out_shape(n, h, w)
        st.update(L=L, gdn=gd, x=codes(g, n, h, w, GDN_C, 0.5, scale(0.5)), z=i8(*shape), y=i8(*shape))
    elif kind == "synthesis":
        T = synthesis_model()
        st.update(T=T, x=codes(g, n, h, w, 320, 3.0, S_LATENT), op=i8(n, h, w, 320), outs=[])
        for t in T:
            st["outs"].append(i8(*t.out_shape(n, h, w)))
            h, w = 2 * h, 2 * w
    elif kind == "subpixel":
        st.update(L=subpixel_model(), x=codes(g, n, h, w, 192, 0.5, scale(0.5)), y=i8(n, 2 * h, 2 * w, 192))
    else:
        L = affine_model()
        st.update(L=L, x=halves(g, n, h, w, 192, 1.0), op=torch.empty((n, h, w, 192), dtype=torch.int16, device=DEV),
                  params=torch.empty(2, dtype=torch.float32, device=DEV),
                  workspace=torch.empty(64, dtype=torch.uint8, device=DEV),
                  y=torch.empty(L.out_shape(n, h, w), dtype=torch.float32, device=DEV))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "f16_layer":
        return hatq.layer(st["x"], hatq.IN_F16, 1.0, st["P"], y=st["y"], scratch=st["scratch"])
    if kind == "i8_layer":
        return hatq.layer(st["x"], hatq.IN_I8, S_ACT, st["P"], y=st["y"], scratch=st["scratch"])
    if kind == "analysis":
        return st["chain"].forward(st["x"], hatq.IN_I8, S_IMAGE, st["outs"], st["scratch"])
    if kind == "entropy":
        return [ch.forward(x, hatq.IN_I8, S_LATENT, outs, scratch)[-1] for ch, x, outs, scratch in st["runs"]]
    if kind == "quantize":
        x_kind = hatq.IN_I8 if case["dtype"] == "i8" else hatq.IN_F16
        if case["dynamic"]:
            return hatq.quantize_act(st["x"], x_kind, S_ACT, case["hb"], 0.0, y=st["y"], s_used=st["s_used"],
                                     workspace=st["workspace"])
        return hatq.quantize_act(st["x"], x_kind, S_ACT, case["hb"], scale(1.5), y=st["y"])
    if kind == "gdn_layer":
        hatq.conv2d_i8(st["x"], st["L"], y=st["z"])
        return st["z"], hatq.gdn(st["z"], st["gdn"], y=st["y"])
    if kind == "synthesis":
        cur = hatq.quantize_act(st["x"], hatq.IN_I8, S_LATENT, 64, scale(3.0), y=st["op"])
        for T, y in zip(st["T"], st["outs"]):
            cur = hatq.conv_transpose2d_i8(cur, T, y=y)
        return st["outs"]
    if kind == "subpixel":
        return hatq.conv2d_i8_subpixel(st["x"], st["L"], 2, y=st["y"])
    op, params = hatq.quantize_act_affine(st["x"], 64, y=st["op"], params=st["params"], workspace=st["workspace"])
    return op, params, hatq.conv2d_affine(op, st["L"], params, y=st["y"])


# ------------------------------------------------------------------ work, tolerance, 64-bit results

def layer_work(L, n, h, w, in_bytes=1, out_bytes=1):
    ho, wo = L.out_hw(h, w)
    return (n * h * w * L.c_in * in_bytes + n * ho * wo * L.c_out * out_bytes + L.weight_bytes(), 2 * L.macs(n, h, w))


def chain_work(layers, n, h, w):
    by = fl = 0
    for L in layers:
        b, f = layer_work(L, n, h, w)
        by, fl = by + b, fl + f
        h, w = L.out_hw(h, w)
    return by, fl


def work(case):
    kind, n, h, w = case["kind"], case["n"], case["h"], case["w"]
    if kind == "f16_layer":
        by, fl = layer_work(layer(case["c"], case["c"], 1, 1, "DH", "none"), n, h, w, 2, 4)
    elif kind == "i8_layer":
        by, fl = layer_work(i8_layer(case), n, h, w)
    elif kind == "analysis":
        by, fl = chain_work(ANALYSIS, n, h, w)
    elif kind == "entropy":
        parts = [chain_work(c, n, h, w) for c in entropy_layers()]
        by, fl = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "quantize":
        elems = n * h * w * case["c"]
        by, fl = elems * (2 if case["dtype"] == "i8" else 3), elems * int(math.log2(case["hb"]))
    elif kind == "gdn_layer":
        L = layer(GDN_C, GDN_C, 5, 2, "DH", "none")
        by, fl = layer_work(L, n, h, w)
        ho, wo = L.out_hw(h, w)
        by, fl = by + n * ho * wo * GDN_C, fl + 2 * n * ho * wo * GDN_C * GDN_C
    elif kind == "synthesis":
        by, fl = n * h * w * 320, 0
        for ci, co, _ in SYNTHESIS:
            by, fl = by + n * h * w * (ci + 4 * co) + 25 * ci * co, fl + 2 * n * h * w * 25 * ci * co
            h, w = 2 * h, 2 * w
    elif kind == "subpixel":
        by, fl = layer_work(SUBPIXEL, n, h, w)
    else:
        by, fl = layer_work(AFFINE, n, h, w, 2, 4)
        by += n * h * w * 192 * 2
    return {"bytes": int(by), "flops": int(fl)}


def tolerance(case):
    # integer codes from integers are exact; codes from fp16 values are rounded from 32-bit transforms, where
    # another order of the sums moves a few values across a rounding boundary by one code
    if case["kind"] == "f16_layer":
        return {"rel": 2e-4, "max": 0.05}
    if case["kind"] == "affine":
        return {"rel": 2e-4, "max": 0.05, "differ": 1e-3}
    if case["kind"] == "quantize" and case["dtype"] == "f16":
        return {"rel": 1e-6, "differ": 1e-3}
    return "exact"


def hadamard(hb):
    h = torch.ones((1, 1), dtype=torch.float64, device=DEV)
    while h.shape[0] < hb:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h / math.sqrt(hb)


def transform64(x, hb):
    return (x.double().reshape(*x.shape[:-1], -1, hb) @ hadamard(hb)).reshape(x.shape)


def weights64(L, seed):
    """(weight codes [c_out, k, k, c_in], their scale per channel, bias) of a DH layer."""
    w, b = weights(L.c_out, L.k, L.c_in, seed)
    w = transform64(torch.from_numpy(w).to(DEV), L.hb_in)
    s = w.abs().amax(dim=(1, 2, 3)) / 127.0
    return torch.round(w / s[:, None, None, None]), s, torch.from_numpy(b).to(DEV).double()


def conv64(x, w, L):
    """NHWC convolution of a DH layer, tap by tap."""
    n, h, wd, _ = x.shape
    ho, wo = L.out_hw(h, wd)
    xp = torch.nn.functional.pad(x, (0, 0, L.pad, L.pad, L.pad, L.pad))
    y = torch.zeros((n, ho, wo, L.c_out), dtype=torch.float64, device=DEV)
    for ky in range(L.k):
        for kx in range(L.k):
            y += xp[:, ky:ky + (ho - 1) * L.stride + 1:L.stride, kx:kx + (wo - 1) * L.stride + 1:L.stride] @ w[:, ky, kx].T
    return y


def exact(case, seed):
    if case["kind"] == "f16_layer":
        st, c = prepare(case, seed), case["c"]
        L = layer(c, c, 1, 1, "DH", "none")
        w, s_w, b = weights64(L, 300)
        q = torch.clamp(torch.round(transform64(st["x"], L.hb_in) / F16_S_X), -127, 127)
        s_a = F16_S_X * s_w
        return (conv64(q, w, L) + torch.round(b / s_a)) * s_a
    if case["kind"] == "affine":
        st = prepare(case, seed)
        w, s_w, b = weights64(AFFINE, 800)
        v = transform64(st["x"], AFFINE.hb_in)
        lo, hi = min(v.min().item(), 0.0), max(v.max().item(), 0.0)
        s = (hi - lo) / 255.0
        z = min(max(round(-lo / s), 0), 255)
        q = torch.clamp(torch.round(v / s) + z, 0, 255) - z
        y = torch.relu(conv64(q, w, AFFINE) * (s * s_w) + b)
        return None, torch.tensor([s, float(z)], dtype=torch.float64, device=DEV), y
    if case["kind"] == "quantize" and case["dynamic"]:
        # the scale is a computed number; the codes are whole
        v = transform64(prepare(case, seed)["x"], case["hb"]).abs().max()
        return None, (v * (S_ACT if case["dtype"] == "i8" else 1.0) / 127.0).reshape(1)
    return None
