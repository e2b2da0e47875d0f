"""The window convolution (layers with c_in % 16 == 0 and more than one tap) where
its units, K steps, chunks and window offsets can go wrong: channel counts that
do not fill a 64-channel block, 32-channel layers, both strides with odd and
even kernels, several exact chunks per tile with and without 128-wide groups,
ragged outputs. Bit-exact against the oracle; every test also asserts which kernel
and epilogue its sizes take."""
import numpy as np
import pytest

from synth import configs as C
from tests.test_gpu_conv_lean import H, dev, layer_from_codes, run_both  # noqa: F401

pytestmark = pytest.mark.gpu


def takes(H, P, n, h, w, kernel=None, epilogue=None, pair=None, r=0):
    """Asserts the kernel of the call (the window kernel if not said otherwise), its epilogue number
    and whether it runs as CTA pairs."""
    info = H.conv_kernel(P, n, h, w, r)
    assert info.kernel == (H.KERNEL_WINDOW if kernel is None else kernel)
    assert epilogue is None or info.epilogue == epilogue
    assert pair is None or info.pair == pair


def case(H, c_in, c_out, k, stride, hb_next, n, h, w, act="relu", form="DH", lim=127, chunks=None, **kernel):
    rng = np.random.default_rng(c_in * 31 + c_out + k)
    q = rng.integers(-lim, lim + 1, size=(c_out, k, k, c_in))
    q[:, k // 2, k // 2, 0] = 127                            # the channel's scale: the codes stay as drawn
    L, wt = layer_from_codes(q, form, stride, act)
    x = rng.integers(-127, 128, size=(n, h, w, c_in)).astype(np.int8)
    s_y = 0.0002 * lim * np.sqrt(k * k * c_in)
    got, ref, P = run_both(H, L, wt, rng.normal(0, 1, c_out).astype(np.float32), 0.05, s_y, hb_next, x)
    assert np.array_equal(got, ref)
    assert np.mean(np.abs(ref.astype(int)) == 127) < 0.2 and len(np.unique(ref)) > 20
    if chunks is not None:
        units = (c_in + 63) // 64 * (2 if stride == 2 else 1)
        assert -(-units // P.struct.chunk_units) == chunks
    takes(H, P, n, h, w, **kernel)


@pytest.mark.parametrize("c_in", [16, 32, 48, 64, 80, 96, 160, 224])
@pytest.mark.parametrize("k,stride", [(3, 1), (5, 2), (2, 1), (4, 2)])
def test_channel_blocks_and_kernels(H, c_in, k, stride):
    case(H, c_in, 64, k, stride, 64, 2, 19, 21, lim=60)


@pytest.mark.parametrize("c_in,c_out,k,stride,hb_next,chunks", [
    (320, 192, 3, 1, 64, 2), (192, 192, 5, 2, 64, 3), (320, 160, 3, 1, 32, 2), (384, 96, 3, 1, 0, 2),
    (320, 128, 3, 1, 128, 2), (320, 32, 3, 1, 0, 2), (192, 128, 3, 1, 128, 1)])
def test_several_exact_chunks_per_tile(H, c_in, c_out, k, stride, hb_next, chunks):
    """Uniform codes (mean 64): the reduction needs several chunks, drained into registers
    (groups up to 64) or kept in two accumulator regions (128-wide groups). 20 tiles per image,
    so that CTAs of the last layers run several tiles and the regions are reused."""
    epilogue = 2064 if hb_next < 128 else 2128 if chunks == 2 else 1128
    case(H, c_in, c_out, k, stride, hb_next, 9, 64 * stride, 40 * stride, chunks=chunks, epilogue=epilogue,
         pair=int(c_in * k * k // 64 >= 40))


@pytest.mark.parametrize("c_in,chunks", [(256, 2), (320, 2), (576, 3)])
@pytest.mark.parametrize("c_out,images", [(32, 24), (352, 5)])
def test_drained_tiles_with_columns_for_one_warpgroup(H, c_in, chunks, c_out, images):
    """Tiles of 32 columns drained over several chunks: the second epilogue warpgroup has no
    columns of its own and only takes part in the regions' release. Ten tiles per CTA (with and
    without CTA pairs), so each region is handed over many times. The images repeat two base ones."""
    rng = np.random.default_rng(c_in + c_out)
    L, wt = layer_from_codes(rng.integers(-127, 128, size=(c_out, 3, 3, c_in)), "DH", 1, "relu")
    base = rng.integers(-127, 128, size=(2, 64, 40, c_in)).astype(np.int8)
    pick = rng.integers(0, 2, images * 4)
    s_y = 0.0254 * np.sqrt(9 * c_in)
    b = rng.normal(0, 1, c_out).astype(np.float32)
    _, ref, P = run_both(H, L, wt, b, 0.05, s_y, 0, base)
    units = -(-c_in // 64)
    assert -(-units // P.struct.chunk_units) == chunks
    takes(H, P, images * 4, 64, 40, epilogue=2064, pair=int(c_in > 256))
    assert H.conv_kernel(P, images * 4, 64, 40).n_t == 32
    for _ in range(3):
        y = H.conv2d_i8(dev(base[pick]), P)
        H.sync_status()
        assert np.array_equal(y.cpu().numpy(), ref[pick])


@pytest.mark.parametrize("n,h,w", [(2, 33, 17), (21, 64, 40)])     # ragged; more pairs of tiles than CTA pairs
@pytest.mark.parametrize("hb_out,hb_next", [(64, 64), (64, 0), (64, 32)])
def test_output_transform_with_chunks(H, hb_out, hb_next, n, h, w):
    """A WH layer of several chunks: the 64-wide output transform is shared by two warps. The
    images repeat two base ones."""
    rng = np.random.default_rng(hb_next + h)
    L, wt = layer_from_codes(rng.integers(-127, 128, size=(192, 3, 3, 320)), "WH", 1, "relu")
    base = rng.integers(-127, 128, size=(2, h, w, 320)).astype(np.int8)
    pick = np.concatenate([[0, 1], rng.integers(0, 2, n - 2)])
    _, ref, P = run_both(H, L, wt, rng.normal(0, 1, 192).astype(np.float32), 0.05, 0.0254 * np.sqrt(9 * 320), hb_next, base)
    assert np.mean(np.abs(ref.astype(int)) == 127) < 0.2 and len(np.unique(ref)) > 20
    takes(H, P, n, h, w, epilogue=2064, pair=1)
    assert H.conv_kernel(P, n, h, w).chunks == 2
    y = H.conv2d_i8(dev(base[pick]), P)
    H.sync_status()
    assert np.array_equal(y.cpu().numpy(), ref[pick])


@pytest.mark.parametrize("hb_next", [0, 32, 64])
def test_output_transform_with_chunks_in_the_general_kernel(H, hb_next):
    """The same layer on an output that fills 8 x 16 tiles badly."""
    case(H, 320, 192, 3, 1, hb_next, 1, 33, 26, form="WH", chunks=2, kernel=H.KERNEL_GENERAL)


@pytest.mark.parametrize("h,w", [(16, 8), (31, 15), (15, 7), (17, 23), (48, 1), (33, 17)])
def test_ragged_windows(H, h, w):
    case(H, 64, 192, 3, 1, 64, 3, h, w, epilogue=64, pair=0)


@pytest.mark.parametrize("h,w", [(17, 9), (1, 40), (33, 26)])
def test_outputs_that_fill_the_tiles_badly(H, h, w):
    """The other side of the rule: these take the general kernel's lean form."""
    case(H, 64, 192, 3, 1, 64, 3, h, w, kernel=H.KERNEL_LEAN, epilogue=64)


@pytest.mark.parametrize("c_out,form", [(256, "DH"), (192, "WH"), (768, "DH")])
@pytest.mark.parametrize("h,w", [(33, 26), (16, 8), (17, 5), (33, 17), (100, 36)])
def test_subpixel_stores(H, c_out, form, h, w):
    """The factor-2 rearrangement in the epilogue's stores, at ragged tile edges."""
    from oracle import hatq_oracle as O
    from tests.test_gpu_conv_lean import dev
    rng = np.random.default_rng(c_out + h)
    L, wt = layer_from_codes(rng.integers(-60, 61, size=(c_out, 3, 3, 64)), form, 1, "relu")
    x = rng.integers(-127, 128, size=(3, h, w, 64)).astype(np.int8)
    b = rng.normal(0, 1, c_out).astype(np.float32)
    P = H.prepare_weights(H.desc_from_spec(L), wt, b, 0.05, 0.3, L.act, 0, False)
    if (h, w) == (33, 26):
        takes(H, P, 3, h, w, kernel=H.KERNEL_GENERAL, r=2)
    else:
        takes(H, P, 3, h, w, epilogue=3064, r=2)
    y = H.conv2d_i8_subpixel(dev(x), P, 2)
    H.sync_status()
    p = O.prepare_layer(wt, b, L.form, L.hb_in, L.hb_out, 0.05, 0.3, L.act, 0, False, 1, 1)
    assert np.array_equal(y.cpu().numpy(), O.depth_to_space(O.conv_layer(x, p), 2))


@pytest.mark.parametrize("c_out,form,hb_next", [(192, "DH", 64), (96, "DH", 32), (128, "WH", 64), (96, "DH", 0)])
@pytest.mark.parametrize("act", ["silu", "gelu"])
@pytest.mark.parametrize("n,h,w", [(3, 33, 26), (3, 33, 17), (9, 63, 39)])
def test_general_transition(H, c_out, form, hb_next, act, n, h, w):
    """SiLU / GELU through the table, both group widths, several tiles with ragged edges; the
    first size takes the general kernel, the last has more tiles than CTAs."""
    from oracle import hatq_oracle as O
    from tests.test_gpu_conv_lean import dev
    rng = np.random.default_rng(c_out + hb_next)
    L, wt = layer_from_codes(rng.integers(-60, 61, size=(c_out, 3, 3, 64)), form, 1, act)
    x = rng.integers(-127, 128, size=(n, h, w, 64)).astype(np.int8)
    s_z, s_u, s_y = (float(np.float32(v)) for v in (0.2, 0.15, 0.3))
    P = H.prepare_weights(H.desc_from_spec(L), wt, None, 0.05, s_y, act, hb_next, s_z=s_z, s_u=s_u)
    if (h, w) == (33, 26):
        takes(H, P, n, h, w, kernel=H.KERNEL_GENERAL)
    else:
        takes(H, P, n, h, w, epilogue=4064 if c_out % 64 == 0 else 4032)
    y = H.conv2d_i8(dev(x), P)
    H.sync_status()
    p = O.prepare_layer(wt, None, L.form, L.hb_in, L.hb_out, 0.05, s_y, act, hb_next, False, 1, 1, s_z=s_z, s_u=s_u)
    ref = O.conv_layer(x, p)
    assert np.array_equal(y.cpu().numpy(), ref)
    assert len(np.unique(ref)) > 20


@pytest.mark.parametrize("n,h,w", [(1, 9, 7), (1, 16, 24), (3, 16, 8), (5, 33, 17)])
@pytest.mark.parametrize("c_out,hb_next", [(192, 64), (128, 128), (32, 0)])
def test_pairs_with_odd_tiles(H, n, h, w, c_out, hb_next):
    """45 weight blocks (CTA pairs), with one M tile and other odd numbers of them: the last pair's
    second tile lies past the last image. Small codes, so that one chunk holds the reduction, and
    uniform ones, so that it takes two."""
    one, two = {64: (64, 2064), 128: (1128, 2128), 0: (32, 2064)}[hb_next]
    case(H, 320, c_out, 3, 1, hb_next, n, h, w, lim=40, epilogue=one, pair=1)
    case(H, 320, c_out, 3, 1, hb_next, n, h, w, chunks=2, epilogue=two, pair=1)


@pytest.mark.parametrize("h,w", [(16, 24), (67, 131)])
def test_dependent_launches_back_to_back(H, h, w):
    """Kernels whose CTAs may be placed before their predecessor has ended: five dependent layers
    of the general, window and GDN kernels, queued many times without a host wait, eagerly and from
    a captured graph; every run's codes equal the first ones, which were waited for one by one."""
    import torch
    rng = np.random.default_rng(h)
    layers, s_x, std = [], 0.05, 0.05 * 35
    for k in (3, 1, 5, 3):
        std *= 0.05 * 8 * k * 0.7
        s_y = float(np.float32(std * 5 / 127))
        L = C.layer("t", 64, 64, k, 1, k // 2, "DH", "relu", hb_in=64)
        wts = (rng.standard_normal((64, k, k, 64)) * 0.05).astype(np.float32)
        layers.append(H.prepare_weights(H.desc_from_spec(L), wts, None, s_x, s_y, "relu", 64))
        s_x = s_y
    gdn = H.prepare_gdn(64, 0.5 + rng.random(64), np.abs(rng.standard_normal((64, 64))) * 0.01, 0.04, 0.02, False, 0.05, 64)
    x = dev(rng.integers(-60, 61, size=(2, h, w, 64)).astype(np.int8))
    bufs = [torch.empty_like(x) for _ in range(5)]

    def run(wait=False):
        cur = x
        for P, y in zip(layers + [None], bufs):
            H.gdn(cur, gdn, y=y) if P is None else H.conv2d_i8(cur, P, y=y)
            if wait:
                H.sync_status()
            cur = y

    run(wait=True)
    ref = [b.clone() for b in bufs]
    assert all(len(torch.unique(b)) > 10 for b in ref)
    for _ in range(20):
        for b in bufs:
            b.zero_()
        run()
        run()
        H.sync_status()
        assert all(torch.equal(a, b) for a, b in zip(bufs, ref))
    graph = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        run()
    for b in bufs:
        b.zero_()
    for _ in range(10):
        graph.replay()
    H.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(bufs, ref))
