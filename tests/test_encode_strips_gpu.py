"""Frame encoder (Section 2) at the edges of its strip kernel: widths around a
lane's 8 pixels and a strip's 240 columns, short frames, every window size,
unaligned frames and odd strides, extreme images and offsets.  Integer
arithmetic throughout, so the comparison with the oracle is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1608_01966_gb300 as spg  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(frames, reduce, block, offset, lead=0, pad=0):
    n, H, W = frames.shape[:3]
    ch = 3 if frames.ndim == 4 else 1
    e = spg.sp_encoder_create(spg.sp_encoder_config_init(src_w=W, src_h=H, channels=ch,
                                                         reduce=reduce, block=block,
                                                         offset=offset))
    info = spg.sp_encoder_get_info(e)
    fb, words = info["src_bytes"], info["out_words"]
    stride = fb + pad
    buf = np.full(lead + n * stride, 0xA5, np.uint8)
    for t in range(n):
        buf[lead + t * stride:lead + t * stride + fb] = frames[t].reshape(-1)
    d = torch.from_numpy(buf).cuda()
    bits = torch.full((n, words + 1), -1, dtype=torch.int32, device="cuda")
    spg.sp_encode_device(e, d[lead:], n, stride, bits, words + 1, torch.cuda.current_stream())
    torch.cuda.synchronize()
    got = bits.cpu().numpy().view(np.uint32)
    spg.sp_encoder_destroy(e)
    assert (got[:, words] == 0xFFFFFFFF).all(), "wrote past the encoded frame"
    got = np.unpackbits(np.ascontiguousarray(got[:, :words]).view(np.uint8), bitorder="little")
    got = got.reshape(n, -1)
    want = np.stack([oracle.encode(f, reduce, block, offset).reshape(-1) for f in frames])
    nb = want.shape[1]
    np.testing.assert_array_equal(got[:, :nb], want)
    assert not got[:, nb:].any(), "unused high bits of the last word must be zero"


def _random(n, H, W, ch, seed):
    s = (n, H, W, 3) if ch == 3 else (n, H, W)
    return np.random.default_rng(seed).integers(0, 256, s, dtype=np.uint8)


@pytest.mark.parametrize("W", [8, 9, 15, 16, 232, 239, 240, 241, 248, 249, 472, 480, 487])
@pytest.mark.parametrize("ch", [1, 3])
def test_widths(W, ch):
    _check(_random(2, 37, W, ch, W), 1, 11, 2)
    _check(_random(2, 23, 2 * W + W % 2, ch, W + 1), 2, 7, -1)


@pytest.mark.parametrize("block", [3, 5, 7, 9, 11, 13])
@pytest.mark.parametrize("H", [1, 2, 5, 13, 64])
def test_windows_and_heights(block, H):
    _check(_random(1, H, 264, 3, block + H), 1, block, 0)
    _check(_random(1, 2 * H, 250, 1, block), 2, block, 3)


@pytest.mark.parametrize("lead", range(8))
@pytest.mark.parametrize("pad", [0, 1, 6, 8])
def test_unaligned_frames(lead, pad):
    """Frames at every byte of a word, strides that move them from frame to
    frame, the last byte of the buffer being the last pixel's."""
    _check(_random(3, 11, 24, 3, lead), 1, 5, 1, lead, pad)
    _check(_random(3, 12, 50, 1, lead), 2, 3, 0, lead, pad)


@pytest.mark.parametrize("block", [3, 9, 11, 13])
@pytest.mark.parametrize("offset", [-1000, -256, -255, -1, 0, 1, 255, 256, 1000])
def test_extreme_images_and_offsets(block, offset):
    """All-white frames give the largest sums there are, checkerboards and
    single pixels the largest differences."""
    f = np.zeros((4, 40, 256), np.uint8)
    f[0] = 255
    f[1, ::2, ::2] = 255
    f[1, 1::2, 1::2] = 255
    f[2, 20, 128] = 255
    f[3, :, 100:] = 255
    _check(f, 1, block, offset)


def test_many_frames_fill_several_waves():
    _check(_random(40, 70, 1000, 1, 3), 1, 11, 2)
