"""The window convolution (layers with c_in % 16 == 0 and more than one tap) where
its units, K steps, chunks and window offsets can go wrong: channel counts that
do not fill a 64-channel block, 32-channel layers, both strides with odd and
even kernels, several exact chunks per tile with and without 128-wide groups,
ragged outputs. Bit-exact against the oracle."""
import numpy as np
import pytest

from tests.test_gpu_conv_lean import H, layer_from_codes, run_both  # noqa: F401

pytestmark = pytest.mark.gpu


def case(H, c_in, c_out, k, stride, hb_next, n, h, w, act="relu", form="DH", lim=127, chunks=None):
    rng = np.random.default_rng(c_in * 31 + c_out + k)
    L, wt = layer_from_codes(rng.integers(-lim, lim + 1, size=(c_out, k, k, c_in)), form, stride, act)
    x = rng.integers(-127, 128, size=(n, h, w, c_in)).astype(np.int8)
    s_y = 0.0002 * lim * np.sqrt(k * k * c_in)
    got, ref, P = run_both(H, L, wt, rng.normal(0, 1, c_out).astype(np.float32), 0.05, s_y, hb_next, x)
    assert np.array_equal(got, ref)
    assert np.mean(np.abs(ref.astype(int)) == 127) < 0.2 and len(np.unique(ref)) > 20
    if chunks is not None:
        units = (c_in + 63) // 64 * (2 if stride == 2 else 1)
        assert -(-units // P.struct.chunk_units) == chunks


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
    case(H, c_in, c_out, k, stride, hb_next, 9, 64 * stride, 40 * stride, chunks=chunks)


@pytest.mark.parametrize("hb_out,hb_next", [(64, 64), (64, 0), (64, 32)])
def test_output_transform_with_chunks(H, hb_out, hb_next):
    """A WH layer of several chunks: the 64-wide output transform is shared by two warps."""
    case(H, 320, 192, 3, 1, hb_next, 1, 33, 26, form="WH", chunks=2)


@pytest.mark.parametrize("h,w", [(16, 8), (17, 9), (15, 7), (1, 40), (48, 1)])
def test_ragged_windows(H, h, w):
    case(H, 64, 192, 3, 1, 64, 3, h, w)
