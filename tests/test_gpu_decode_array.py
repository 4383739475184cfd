"""hm_codec_decode on arrays: the block kernel (arrays that start on a 16-byte
boundary) equals the byte-wise kernel (the same codes one byte further) bit for
bit, for random codes of every header the encoders can write -- AFLP exponents
beyond 52, FPX e8 zeros, denormals, infinities and NaNs included -- and sizes
around a block of 2048 values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HEADERS = ([(B, 0, 8, 8 * B - 9) for B in (2, 3, 4)] + [(B, 1, 11, 8 * B - 12) for B in (5, 6, 7, 8)] + [(8, 3, 11, 52)] +
           [(B, 2, e, 8 * B - 1 - e) for B in range(1, 8) for e in (1, 2, 5, 6, 10) if 1 <= 8 * B - 1 - e <= 52])


@pytest.mark.parametrize("n", [1, 7, 2047, 2048, 2049, 9001])
def test_block_decode_equals_bytewise(n):
    from paper_2405_03456_gb300 import build, hm
    build.build()
    rng = np.random.default_rng(n)
    for B, fmt, e, m in HEADERS:
        codes = rng.integers(0, 256, n * B, dtype=np.uint8)
        codes[: min(n, 3) * B] = 0
        if fmt == 0 and n > 8:   # an infinity / a NaN
            codes[7 * B:8 * B] = [0] * (B - 2) + [0x80, 0x7f]
            codes[8 * B:9 * B] = [1] * (B - 2) + [0x80, 0xff]
        hdr = {"B": B, "fmt": fmt, "e": e, "m": m, "vmin": 0.7234567891234567 * 2.0 ** -9 if fmt == 2 else 1.0}
        buf = torch.zeros(n * B + 32, dtype=torch.uint8, device="cuda")
        assert buf.data_ptr() % 16 == 0
        outs = []
        for off in (0, 1):
            buf[off:off + n * B] = torch.from_numpy(codes).cuda()
            out = torch.full((n + 1,), -7.0, dtype=torch.float64, device="cuda")
            hm.hm_codec_decode(buf.data_ptr() + off, n, hdr, out.data_ptr())
            torch.cuda.synchronize()
            outs.append(out.cpu().numpy())
        assert np.array_equal(outs[0].view(np.uint64), outs[1].view(np.uint64)), (B, fmt, e, m)
        assert outs[0][n] == -7.0
