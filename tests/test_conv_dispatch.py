"""Which kernel a convolution call takes (hatq_conv_kernel), on the host alone: the prepared
structs are filled by hand, as the query reads no device memory."""
import numpy as np
import pytest

from paper_2608_01653_gb300 import hatq as H


def struct(c_in, c_out, k=3, stride=1, form="DH", hb_out=0, hb_next=0, act="none", out_f32=False, chunk_kb=1 << 14,
           chunk_units=1 << 10, kw=None, pad=None):
    """A prepared layer's struct whose weight codes are small enough for any chunk length asked for."""
    hb_in = 0
    if form == "DH":
        hb_in = next(h for h in (64, 32, 16) if c_in % h == 0)
    kw = k if kw is None else kw
    d = H.make_desc(c_in, c_out, k, stride, min(k, kw) // 2 if pad is None else pad, form, hb_in=hb_in, hb_out=hb_out, kw=kw)
    s = H.PreparedStruct()
    s.d = d
    s.act, s.hb_next, s.out_f32 = H._ACTS[act], hb_next, int(out_f32)
    s.k_pad = H.prepared_sizes(d)[0] // c_out
    s.gather = int(c_in % 16 != 0)
    s.chunk_kb, s.chunk_units = chunk_kb, chunk_units
    return s


def route(s, n, h, w, r=0):
    i = H.conv_kernel(s, n, h, w, r)
    return i.kernel, i.epilogue, i.pair


G, LEAN, WIN = H.KERNEL_GENERAL, H.KERNEL_LEAN, H.KERNEL_WINDOW


@pytest.mark.parametrize("kw,size,expect", [
    (dict(c_in=64, c_out=192, hb_next=64), (1, 64, 40), (WIN, 64, 0)),
    (dict(c_in=64, c_out=96, hb_next=32), (1, 64, 40), (WIN, 32, 0)),
    (dict(c_in=320, c_out=128, hb_next=128), (1, 64, 40), (WIN, 1128, 1)),
    (dict(c_in=320, c_out=128, hb_next=128, chunk_units=3), (1, 64, 40), (WIN, 2128, 1)),
    (dict(c_in=320, c_out=128, hb_next=128, chunk_units=2, chunk_kb=16), (1, 64, 40), (G, 0, 0)),   # three chunks of 128 columns
    (dict(c_in=320, c_out=192, hb_next=64, chunk_units=3), (1, 64, 40), (WIN, 2064, 1)),
    (dict(c_in=320, c_out=224, hb_next=32, chunk_units=3, chunk_kb=16), (1, 64, 40), (G, 0, 0)),    # drains hold 192 columns
    (dict(c_in=64, c_out=192, hb_next=64, chunk_units=0, chunk_kb=0), (1, 64, 40), (LEAN, 64, 0)),  # codes not known
    (dict(c_in=64, c_out=192, k=5, hb_next=64, chunk_units=0, chunk_kb=0), (1, 64, 40), (G, 0, 0)),
    (dict(c_in=64, c_out=192, k=1, hb_next=64), (1, 64, 40), (LEAN, 64, 0)),                        # one tap
    (dict(c_in=3, c_out=192, k=5, form="WH", hb_out=64), (1, 64, 40), (LEAN, 64, 0)),               # small channels
    (dict(c_in=64, c_out=192, hb_next=64), (1, 33, 17), (WIN, 64, 0)),
    (dict(c_in=64, c_out=192, hb_next=64), (1, 33, 26), (LEAN, 64, 0)),     # 12 tiles of 8 x 16 where 9 of 32 x 4 do
    (dict(c_in=64, c_out=192, hb_next=64), (1, 1, 40), (LEAN, 64, 0)),
    (dict(c_in=64, c_out=192, act="silu", hb_next=64), (1, 64, 40), (WIN, 4064, 0)),
    (dict(c_in=64, c_out=96, act="gelu", hb_next=32), (1, 64, 40), (WIN, 4032, 0)),
    (dict(c_in=128, c_out=192, act="gelu", hb_next=64, chunk_units=1), (1, 64, 40), (G, 0, 0)),
    (dict(c_in=64, c_out=192, out_f32=True), (1, 64, 40), (G, 0, 0)),
    (dict(c_in=64, c_out=64, k=16, kw=4, pad=0), (1, 64, 40), (WIN, 32, 1)),                        # 64 taps
    (dict(c_in=64, c_out=64, k=13, kw=5, pad=0), (1, 64, 40), (LEAN, 32, 0)),                       # 65 taps
])
def test_kernel_of_a_layer(kw, size, expect):
    assert route(struct(**kw), *size) == expect


@pytest.mark.parametrize("act,k,counts", [("silu", 3, {1: 2, 12: 2, 13: 1, 102: 1}), ("relu", 3, {1: 2, 13: 2, 101: 2, 102: 1}),
                                          ("relu", 5, {1: 5, 12: 5, 13: 1})])
def test_few_tiles_per_cta_keep_both_warpgroups(act, k, counts):
    """The int64 epilogue of one long chunk is one warpgroup's; with few tiles per CTA the general chunk
    length stays, and both warpgroups drain and finish a tile."""
    s = struct(192, 192, k, hb_next=64, act=act, chunk_units=0)
    s.out_f16 = int(act == "relu")
    for n, chunks in counts.items():                                 # 12 tiles of 16 x 96 pixels per image
        i = H.conv_kernel(s, n, 16, 96)
        assert (i.kernel, i.chunks) == (G, chunks), n
    assert H.conv_kernel(struct(192, 192, out_f32=True), 1, 16, 96).chunks == 1


@pytest.mark.parametrize("c_out,r,size,expect", [(256, 2, (3, 64, 40), (WIN, 3064, 0)), (256, 2, (3, 33, 26), (G, 0, 0)),
                                                 (64, 2, (3, 64, 40), (WIN, 3064, 0)), (288, 3, (3, 64, 40), None)])
def test_kernel_of_a_subpixel_layer(c_out, r, size, expect):
    s = struct(64, c_out)
    if expect is None:                                       # tiles of 96 columns are not whole groups of 144
        with pytest.raises(H.HatqError) as e:
            H.conv_kernel(s, *size, r)
        assert e.value.status == H.ERR_UNSUPPORTED
    else:
        assert route(s, *size, r) == expect


def test_query_checks_its_arguments():
    s = struct(64, 64)
    assert H.conv_kernel(s, 0, 8, 8).kernel == H.KERNEL_NONE
    for bad in ((1, 0, 8, 0), (1, 8, 8, 1), (1, 8, 8, 5), (-1, 8, 8, 0)):
        with pytest.raises(H.HatqError):
            H.conv_kernel(s, *bad)
    with pytest.raises(H.HatqError):
        H.conv_kernel(H.PreparedStruct(), 1, 8, 8)
    assert H.load().hatq_conv_kernel(None, 1, 8, 8, 0, None) == H.ERR_INVALID_ARG


def test_plans_stay_within_the_documented_limits():
    """Random layers and sizes: two stages or more, shared memory within a CTA's, chunks of whole
    stages, accumulators and operand within 512 tensor-memory columns."""
    rng = np.random.default_rng(5)
    seen = set()
    for _ in range(3000):
        c_in = int(rng.choice([3, 16, 32, 48, 64, 96, 160, 192, 320, 640]))
        c_out = int(rng.choice([32, 64, 96, 128, 192, 320, 640, 352, 1024, 9216]))
        k, stride = int(rng.integers(1, 6)), int(rng.integers(1, 3))
        hb = int(rng.choice([h for h in (0, 16, 32, 64, 128) if h == 0 or c_out % h == 0]))
        wh = c_in % 16 != 0 or rng.random() < 0.3
        hb_out = int(rng.choice([h for h in (16, 32, 64, 128) if c_out % h == 0])) if wh else 0
        s = struct(c_in, c_out, k, stride, "WH" if wh else "DH", hb_out, hb, str(rng.choice(["none", "relu"])),
                   chunk_kb=int(rng.choice([0, 16, 20, 1 << 14])), chunk_units=int(rng.integers(0, 8)))
        try:
            i = H.conv_kernel(s, int(rng.integers(1, 4)), *(int(v) for v in rng.integers(5, 200, 2)))
        except H.HatqError as e:
            assert e.status == H.ERR_UNSUPPORTED
            continue
        seen.add((i.kernel, i.epilogue, i.pair))
        assert i.stages >= 2 and i.blocks >= 1 and 0 < i.smem_bytes <= 227 * 1024 - 1024
        assert c_out % i.n_t == 0 and i.n_t <= 224
        if i.kernel == WIN:
            assert (4 if i.epilogue == 2128 else 2) * i.n_t <= 512 and 2 <= i.stages <= 8
            assert i.chunks == 1 or i.epilogue in (2064, 2128)
        else:
            assert i.blocks in (1, 2, 4) and (i.kernel == G or i.chunks == 1)
    assert {k for k, _, _ in seen} == {G, LEAN, WIN} and {e for k, e, _ in seen if k == WIN} >= {32, 64, 1128, 2064, 2128}


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("hb_next", [0, 64, 128])
def test_wide_layers_are_taken_wherever_a_tile_fits(hb_next, k):
    """The constants of a wide layer (16 bytes per output channel) leave little shared memory. Every
    layer for which two single-block stages fit beside the general epilogue's output tile is accepted,
    whether or not the lean kernel's fixed staging fits there."""
    G_ = max(32, hb_next)
    lean = general = 0
    for c_out in range(8192, 12288 + 1, 128 if hb_next == 128 else 64):
        n_t = next(t for t in range(224, 0, -16) if t % G_ == 0 and c_out % t == 0)
        budget = 226 * 1024 - (1024 + 8 * 37 + 16 + 128 + 16 * c_out) - (1 if G_ == 128 else 2) * 128 * (n_t + 16)
        fits = budget // (n_t * 128 + 8192) >= 2
        try:
            i = H.conv_kernel(struct(64, c_out, k, hb_next=hb_next), 1, 16, 8)
        except H.HatqError as e:
            assert not fits and e.status == H.ERR_UNSUPPORTED, c_out
            continue
        lean, general = lean + (i.kernel == LEAN), general + (i.kernel == G)
        assert i.stages >= 2 and i.smem_bytes <= 227 * 1024 - 1024
    assert lean and general
