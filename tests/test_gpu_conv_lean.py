"""The convolution kernels for INT8 codes without further options, at the
places where their epilogue decides: rounding ties at shifts around a word
boundary, ragged output boxes, and every transform group. Bit-exact against
the oracle."""
import numpy as np
import pytest

from oracle import hatq_oracle as O
from synth import configs as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2608_01653_gb300 import hatq
    hatq.load()
    return hatq


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def layer_from_codes(q, form, stride, act):
    """A layer whose weight codes are q [c_out, k, k, c_in] at scale 2^-10 (blocks of 4 and
    64 have exact square roots, so W and its transform are exact)."""
    co, k, _, ci = q.shape
    L = C.layer("t", ci, co, k, stride, k // 2, form, act, hb_in=4 if form == "DH" else None,
                hb_out=64 if form == "WH" else None)
    if form == "DH":
        w = O.transform_real(q.astype(np.float64), 4)
    else:
        w = np.moveaxis(O.transform_real(np.moveaxis(q.astype(np.float64), 0, -1), 64), -1, 0)
    return L, (w * 2.0 ** -10).astype(np.float32)


def run_both(H, L, w, b, s_x, s_y, hb_next, x):
    P = H.prepare_weights(H.desc_from_spec(L), w, b, s_x, s_y, L.act, hb_next, False)
    y = H.conv2d_i8(dev(x), P)
    H.sync_status()
    p = O.prepare_layer(w, b, L.form, L.hb_in, L.hb_out, s_x, s_y, L.act, hb_next, False, L.stride, L.pad)
    return y.cpu().numpy(), O.conv_layer(x, p), P


@pytest.mark.parametrize("shift", [30, 31, 32, 33, 36])
@pytest.mark.parametrize("c_out,form,hb_next,act", [(64, "DH", 0, "none"), (192, "DH", 64, "relu"), (224, "DH", 32, "none"),
                                                    (128, "DH", 128, "relu"), (64, "WH", 64, "relu"), (32, "DH", 0, "relu")])
def test_power_of_two_scales_round_ties_to_even(H, c_out, form, hb_next, act, shift):
    """M = 2^30 for every channel, so M a / 2^n has ties whatever n is: at n <= 32 the half lies
    in the low word, above it the low word of a tie is zero."""
    rng = np.random.default_rng(shift + c_out)
    q = rng.integers(-2, 3, size=(c_out, 3, 3, 64))
    q[:, 1, 1, 0] = 127                                    # the channel's scale
    L, w = layer_from_codes(q, form, 1, act)
    x = rng.integers(-3, 4, size=(2, 9, 37, 64)).astype(np.int8)
    x[..., 0] = rng.integers(-1, 2, size=(2, 9, 37)) * (rng.random((2, 9, 37)) < 0.2)
    alpha = (8.0 if form == "WH" else 1.0) * np.sqrt(hb_next if hb_next else 1)
    s_y = float(np.float32(2.0 ** -10 * 2.0 ** (shift - 30) / alpha))
    got, ref, P = run_both(H, L, w, np.zeros(c_out, np.float32), 1.0, s_y, hb_next, x)
    assert np.array_equal(got, ref)
    assert H.conv_kernel(P, 2, 9, 37).kernel == H.KERNEL_WINDOW
    if hb_next != 128 and hb_next != 32:                   # alpha is a power of two
        assert P.struct.shift == shift
    assert len(np.unique(ref)) > 3


@pytest.mark.parametrize("c_in,k", [(64, 3), (64, 1), (3, 5)])        # window, general and small-channel kernels
@pytest.mark.parametrize("c_out,hb_next,act", [(64, 64, "none"), (192, 64, "relu"), (32, 32, "none"), (96, 16, "relu")])
def test_biases_that_leave_every_code_uncertain(H, c_in, k, c_out, hb_next, act):
    """Biases along one Walsh function, some ten thousand codes in norm: they meet in one output of
    each block, and the bound of the fp32 estimate, which grows with the norm, sends nearly every
    row to the exact evaluation."""
    rng = np.random.default_rng(c_in + c_out + k)
    form = "WH" if c_in == 3 else "DH"
    hb = 64 if c_out % 64 == 0 else 32
    L = C.layer("t", c_in, c_out, k, 1, k // 2, form, act, hb_in=64 if form == "DH" else None, hb_out=hb if form == "WH" else None)
    w = rng.standard_normal((c_out, k, k, c_in)).astype(np.float32) * 0.05
    x = rng.integers(-60, 61, size=(2, 19, 23, c_in)).astype(np.int8)
    s_y = 0.05 * np.sqrt(c_in * k * k) * 35 * 0.02 * 8 / 40
    sign = 1 - 2 * (np.arange(c_out) & 1)                             # a Walsh function of every block size
    b = (1500 * 8 * s_y * sign).astype(np.float32)
    got, ref, P = run_both(H, L, w, b, 0.02, float(np.float32(s_y)), hb_next, x)
    assert np.array_equal(got, ref)
    assert H.conv_kernel(P, 2, 19, 23).kernel == (H.KERNEL_WINDOW if (c_in, k) == (64, 3) else H.KERNEL_LEAN)
    assert len(np.unique(ref)) > 20


@pytest.mark.parametrize("h,w", [(1, 1), (1, 129), (5, 31), (17, 33), (130, 3), (16, 64)])
@pytest.mark.parametrize("c_out,hb_next", [(192, 64), (96, 32), (128, 128)])
def test_ragged_output_boxes(H, h, w, c_out, hb_next):
    """Output sizes at the edges of the warps' 32-row boxes; two images."""
    rng = np.random.default_rng(h * 1000 + w)
    L, wt = layer_from_codes(rng.integers(-127, 128, size=(c_out, 1, 1, 64)), "DH", 1, "relu")
    x = rng.integers(-127, 128, size=(2, h, w, 64)).astype(np.int8)
    got, ref, P = run_both(H, L, wt, rng.normal(0, 1, c_out).astype(np.float32), 0.05, 0.11, hb_next, x)
    assert np.array_equal(got, ref)
    assert H.conv_kernel(P, 2, h, w).kernel == H.KERNEL_LEAN


@pytest.mark.parametrize("avg,one_chunk", [(120, True), (122, False)])
@pytest.mark.parametrize("sign", [1, -1])
def test_whole_reduction_in_one_exact_chunk(H, avg, one_chunk, sign):
    """1088 weight codes of average magnitude 120: 128 sum |w| stays below 2^24, so the layer takes
    the reduction in one chunk, and with operand codes of -128 and 127 the sums come within 0.4 %
    of 2^24; at 122 they would pass it and the general 1024-long chunk stays. The bias cancels the
    sum, so the output shows its low bits."""
    k = 1088
    q = np.full((32, 1, 1, k), avg)
    q[:, 0, 0, 0] = 127
    s = np.where(np.arange(32) % 2, 1, -1)[:, None, None, None]
    L, w = layer_from_codes(q * s, "DH", 1, "none")
    x = np.full((1, 5, 27, k), -128 if sign < 0 else 127, np.int8)
    x[0, 1:, :, 5] -= 1 * sign
    x[0, 2:, 3:, 7] -= 2 * sign
    x[0, :, 9::2, 1] += np.int8(-sign)
    s_w = 2.0 ** -10
    total = int(np.abs(q[0]).sum()) * (128 if sign < 0 else 127)
    b = (-sign * s[:, 0, 0, 0] * (total - 300) * s_w).astype(np.float32)
    got, ref, P = run_both(H, L, w, b, 1.0, float(np.float32(8 * s_w)), 0, x)
    assert np.array_equal(got, ref)
    assert (P.struct.chunk_kb >= k // 64) == one_chunk
    assert H.conv_kernel(P, 1, 5, 27).kernel == (H.KERNEL_LEAN if one_chunk else H.KERNEL_GENERAL)
    assert len(np.unique(ref)) > 3


@pytest.mark.parametrize("c_out,hb_next", [(9216, 128), (10048, 64), (9696, 32)])
def test_wide_layers_without_room_for_the_lean_staging(H, c_out, hb_next):
    """Their constants leave shared memory for two stages beside the general epilogue's output tile
    only."""
    rng = np.random.default_rng(c_out)
    L, wt = layer_from_codes(rng.integers(-127, 128, size=(c_out, 1, 1, 64)), "DH", 1, "relu")
    x = rng.integers(-127, 128, size=(1, 5, 31, 64)).astype(np.int8)
    got, ref, P = run_both(H, L, wt, rng.normal(0, 1, c_out).astype(np.float32), 0.05, 0.11, hb_next, x)
    assert H.conv_kernel(P, 1, 5, 31).kernel == H.KERNEL_GENERAL
    assert np.array_equal(got, ref)
    assert len(np.unique(ref)) > 20


@pytest.mark.parametrize("c_in,k", [(1088, 1), (128, 3)])              # general and window kernel as prepared
def test_overwritten_weight_codes(H, c_in, k):
    """Codes written over a prepared layer's, with sums beyond the prepared chunk: exact once the
    layer has been told. The bias cancels the sum, so the output shows its low bits."""
    rng = np.random.default_rng(k)
    q = np.full((32, k, k, c_in), 100)
    q[:, 0, 0, 0] = 127
    L, w = layer_from_codes(q, "DH", 1, "none")
    x = np.full((1, 16, 24, c_in), 127, np.int8)
    dec = 1 + 40 // (k * k)
    x[..., 1:dec] -= rng.integers(0, 2, size=(1, 16, 24, dec - 1)).astype(np.int8)
    total, s_w = 127 * 127 * c_in * k * k, 2.0 ** -10
    b = np.full(32, -(total - 4000) * s_w, np.float32)
    P = H.prepare_weights(H.desc_from_spec(L), w, b, 1.0, float(np.float32(80 * s_w)), "none", 0, False)
    assert H.conv_kernel(P, 1, 16, 24).chunks == 1 and total > 2 ** 24
    P.w_i8[P.w_i8 != 0] = 127
    P.w_f16[P.w_f16 != 0] = 127.0
    P.codes_changed()
    assert H.conv_kernel(P, 1, 16, 24).kernel == H.KERNEL_GENERAL
    y = H.conv2d_i8(dev(x), P)
    H.sync_status()
    p = O.prepare_layer(w, b, L.form, L.hb_in, L.hb_out, 1.0, float(np.float32(80 * s_w)), "none", 0, False, L.stride, L.pad)
    p.w_int = np.full_like(p.w_int, 127)
    ref = O.conv_layer(x, p)
    assert np.array_equal(y.cpu().numpy(), ref) and len(np.unique(ref)) > 3
