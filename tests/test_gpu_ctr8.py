"""CTR on 8-byte-aligned buffers: warps that take several tiles, the ragged last
tile, in place and between buffers of different alignment, against the 16-byte
path's result, with the bytes around the output untouched."""
import pytest

from paper_2007_10752_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one warp per CTA with a ragged tile, the widest grid's second pass, its third
SIZES = [1024 * 300 + 1, 1024 * 2500 + 77, 1024 * 5000 + 1023]


@pytest.mark.parametrize("nblocks", SIZES)
@pytest.mark.parametrize("stages", [1, 3])
def test_same_as_16_byte_aligned(cuda_lib, stages, nblocks):
    key, n, ctr0 = synth.key_triple(12), 8 * nblocks, (1 << 32) - nblocks  # to the last counter
    ks = cuda_lib.KeySchedule.des(key[:8]) if stages == 1 else cuda_lib.KeySchedule.from_triple(key)
    src = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")
    synth.fill_device(src, nblocks)
    data = src[:n].clone()
    want = torch.empty_like(data)
    cuda_lib.tdes_ctr_crypt(ks, 5, ctr0, data, want)
    for off_in, off_out in ((8, 8), (0, 24), (8, 16)):
        src[off_in:off_in + n] = data
        dst = torch.full((n + 48,), 0xA5, dtype=torch.uint8, device="cuda")
        cuda_lib.tdes_ctr_crypt(ks, 5, ctr0, src[off_in:off_in + n], dst[off_out:off_out + n])
        assert torch.equal(dst[off_out:off_out + n], want), (off_in, off_out)
        assert bool((dst[:off_out] == 0xA5).all()) and bool((dst[off_out + n:] == 0xA5).all())
    src[8:8 + n] = data
    cuda_lib.tdes_ctr_crypt(ks, 5, ctr0, src[8:8 + n], src[8:8 + n])
    assert torch.equal(src[8:8 + n], want)
