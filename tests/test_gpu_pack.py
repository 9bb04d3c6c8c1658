"""The packing kernels at the sizes and alignments where their vector and byte-wise parts meet: fewer codes than a
group of 16, remainders, more groups than one round of the grid, and pointers aligned for no vector access."""
import numpy as np
import pytest
import torch

from paper_1911_08076_gb300 import ifq, synth

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("kbits", [2, 3, 4])
@pytest.mark.parametrize("n", [4, 12, 16, 4 * 1237, 16 * 1024 + 8, 40 * 1024 * 1024 + 20])
@pytest.mark.parametrize("off_codes,off_packed", [(0, 0), (4, 0), (0, 1), (16, 8), (0, 4)])
def test_pack_and_unpack(kbits, n, off_codes, off_packed):
    fb = synth.field_bits(kbits)
    nb = n * fb // 8
    # bytes above the field are dropped
    raw = torch.from_numpy(np.random.default_rng(n + kbits).integers(0, 256, n, dtype=np.uint8)).cuda()
    codes = torch.empty(off_codes + n, dtype=torch.uint8, device="cuda")[off_codes:]
    codes.copy_(raw)
    buf = torch.full((off_packed + nb + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_codes_kbits(codes, buf[off_packed:], n, kbits)
    want = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    low = raw & ((1 << fb) - 1)
    for i in range(8 // fb):
        want |= low[i::8 // fb] << (fb * i)
    assert torch.equal(buf[off_packed:off_packed + nb], want)
    assert (buf[:off_packed] == 0xA5).all() and (buf[off_packed + nb:] == 0xA5).all()
    back = torch.full((off_codes + n + 16,), 0x5A, dtype=torch.uint8, device="cuda")
    ifq.ifq_unpack_codes_kbits(buf[off_packed:], back[off_codes:], n, kbits)
    assert torch.equal(back[off_codes:off_codes + n], low)
    assert (back[:off_codes] == 0x5A).all() and (back[off_codes + n:] == 0x5A).all()
