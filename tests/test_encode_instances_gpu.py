"""Every instance of the encoder's strip kernel (window, channels, reduction,
aligned rows or not), on sizes that are sure to take it: the rule that picks
the kernel is compiled from its header and asked for every call.  Random and
extreme images, offsets past the range of a difference, frames at every byte
of a word.  Integer arithmetic: the comparison with the oracle is exact."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1608_01966_gb300 as spg  # noqa: E402

pytestmark = pytest.mark.gpu

RULE = """
#include "sp_encode_rule.h"
extern "C" int in_strips(unsigned W, unsigned H, unsigned ch, unsigned f, unsigned block,
                         unsigned n, unsigned long long at, unsigned long long stride, unsigned sms) {
  const unsigned Wr = W / f, Hr = H / f;
  const bool a8 = at % 8 == 0 && stride % 8 == 0 && W * ch % 8 == 0 && Wr % 8 == 0;
  const bool words = at % 4 == 0 && stride % 4 == 0;
  return sp::encode_in_strips({W, ch, f, Wr, Hr, block, n, a8, words, sms}) ? 1 + a8 : 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(RULE)
    csrc = os.path.join(os.path.dirname(spg.__file__), "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", csrc, "-o",
                    str(d / "rule.so"), str(d / "rule.cpp")], check=True)
    fn = ct.CDLL(str(d / "rule.so")).in_strips
    fn.argtypes = [ct.c_uint] * 6 + [ct.c_ulonglong] * 2 + [ct.c_uint]
    return fn


def _check(rule, frames, reduce, block, offset, aligned, lead=0, pad=0):
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
    d = torch.from_numpy(buf).cuda()[lead:]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert rule(W, H, ch, reduce, block, n, d.data_ptr(), stride, sms) == (2 if aligned else 1)
    bits = torch.full((n, words + 1), -1, dtype=torch.int32, device="cuda")
    spg.sp_encode_device(e, d, n, stride, bits, words + 1, torch.cuda.current_stream())
    torch.cuda.synchronize()
    got = bits.cpu().numpy().view(np.uint32)
    spg.sp_encoder_destroy(e)
    assert (got[:, words] == 0xFFFFFFFF).all(), "wrote past the encoded frame"
    got = np.unpackbits(np.ascontiguousarray(got[:, :words]).view(np.uint8), bitorder="little")
    got = got.reshape(n, -1)
    want = np.stack([oracle.encode(f, reduce, block, offset).reshape(-1) for f in frames])
    np.testing.assert_array_equal(got[:, :want.shape[1]], want)
    assert not got[:, want.shape[1]:].any(), "unused high bits of the last word must be zero"


def _widths(reduce, aligned):
    if aligned:
        return [232 * reduce, 240 * reduce, 472 * reduce]
    return [470 * reduce + reduce // 2, 475 * reduce]  # not a multiple of 4; two strips


def _extreme(H, W, ch):
    """All white gives the largest sums, checkerboards and single pixels the
    largest differences."""
    f = np.zeros((5, H, W), np.uint8)
    f[0] = 255
    f[1, ::2, ::2] = 255
    f[1, 1::2, 1::2] = 255
    f[2, H // 2, W // 2] = 255
    f[3, :, W // 2:] = 255
    f[4] = 255
    f[4, H // 3, W // 3:W // 3 + 2] = 0
    return np.repeat(f[..., None], 3, 3) if ch == 3 else f


INSTANCES = [(b, ch, f, a) for b in (3, 5, 7, 9, 11, 13) for ch in (1, 3) for f in (1, 2)
             for a in (True, False)
             if (not a or ch == 3 or f == 1)          # gray halved has one instance
             and (a or ch == 1 or b <= 7)]            # unaligned RGB of tall windows: band kernel


@pytest.mark.parametrize("block,ch,reduce,aligned", INSTANCES)
def test_instance(rule, block, ch, reduce, aligned):
    r = np.random.default_rng(block * 100 + ch * 10 + reduce)
    for W in _widths(reduce, aligned):
        for H, n in ((1, 2), (block // 2, 1), (2 * block + 3, 2), (41, 1)):
            H *= reduce
            shape = (n, H, W) + ((3,) if ch == 3 else ())
            _check(rule, r.integers(0, 256, shape, dtype=np.uint8), reduce, block, 2, aligned)
    f = _extreme(36 * reduce, W, ch)[:2 if ch == 3 and not aligned else 5]
    for offset in (-1000, -256, -255, -1, 0, 1, 255, 256, 1000):
        _check(rule, f, reduce, block, offset, aligned)
    f = _extreme(20 * reduce, W, ch)[2:]
    _check(rule, f, reduce, block, -1, aligned)
    if aligned:
        _check(rule, f, reduce, block, 3, aligned, 8, 8)
        return
    for lead in range(8):
        for pad in (0, 1, 3, 6):
            f = r.integers(0, 256, (2, 9 * reduce, W) + ((3,) if ch == 3 else ()), dtype=np.uint8)
            _check(rule, f, reduce, block, 1, aligned, lead, pad)


def test_calls_of_any_other_size_have_a_kernel():
    """The rule sends no call to an instance that is not compiled."""
    for ch in (1, 3):
        for block in (3, 9, 13):
            for W in (7, 8, 61, 230, 469, 470, 950):
                for reduce in (1, 2, 3):
                    f = np.random.default_rng(W).integers(
                        0, 256, (2, 30, W) + ((3,) if ch == 3 else ()), dtype=np.uint8)
                    e = spg.sp_encoder_create(spg.sp_encoder_config_init(
                        src_w=W, src_h=30, channels=ch, reduce=reduce, block=block, offset=0))
                    words = spg.sp_encoder_get_info(e)["out_words"]
                    bits = torch.zeros((2, words), dtype=torch.int32, device="cuda")
                    d = torch.from_numpy(f.reshape(2, -1)).cuda()
                    spg.sp_encode_device(e, d, 2, d.shape[1], bits, words,
                                         torch.cuda.current_stream())
                    torch.cuda.synchronize()
                    got = np.unpackbits(bits.cpu().numpy().view(np.uint8), axis=1, bitorder="little")
                    for t in range(2):
                        want = oracle.encode(f[t], reduce, block, 0).reshape(-1)
                        np.testing.assert_array_equal(got[t][:len(want)], want)
                    spg.sp_encoder_destroy(e)
