"""The march kernel (narrow pooled first layers on mma.sync f16): codes bit-exact against the CPU oracle at one
pooled pixel, ragged strips of 8 pooled columns, marches that end early, odd paddings and channel counts that fill
no tile of 8, on 8-bit values and on 2-bit codes."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1911_08076_gb300 import ifq, synth

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CASES = [
    # in_bits, n, h, w, cout, pad
    (8, 1, 2, 2, 8, 1), (8, 2, 34, 38, 16, 1), (8, 3, 70, 18, 4, 1), (8, 2, 10, 150, 12, 1), (8, 1, 20, 24, 8, 0),
    (8, 2, 8, 12, 16, 2), (8, 40, 64, 66, 8, 1),
    (0, 1, 2, 2, 8, 1), (0, 2, 34, 38, 16, 1), (0, 3, 70, 18, 32, 1), (0, 2, 10, 150, 8, 1), (0, 40, 64, 66, 16, 1),
]


@pytest.mark.parametrize("case", CASES, ids=[f"b{c[0]}n{c[1]}_{c[2]}x{c[3]}c{c[4]}p{c[5]}" for c in CASES])
@pytest.mark.parametrize("values", ["random", "largest"])
def test_march_matches_oracle(case, values):
    in_bits, n, h, w, cout, pad = case
    cin, top = (4, 255) if in_bits == 8 else (8, 3)
    rng = np.random.default_rng(h * w + cout)
    x = rng.integers(0, top + 1, (n, h, w, cin), dtype=np.uint8)
    wt = np.where(rng.integers(0, 2, (cout, 3, 3, cin)) == 1, 1, -1).astype(np.int8)
    if values == "largest":   # accumulators at both ends of their range
        x[:] = top
        wt[0], wt[1] = 1, -1
    A = O.maxpool_acc(O.conv_acc(x, wt, 1, pad), 2, 2, 0)
    sd = np.sqrt(9 * cin * top * top / 3)
    T = np.sort(rng.normal(0, sd, (cout, 3)), axis=1).astype(np.int32)
    T[0], T[1] = (9 * cin * top - 2, 9 * cin * top - 1, 9 * cin * top), (-9 * cin * top - 1, -9 * cin * top, 2**31 - 1)
    s = np.where(rng.integers(0, 3, cout) == 0, -1, 1).astype(np.int8)
    d = ifq.conv_desc(n, h, w, cin, cout, 3, 1, pad, ifq.IFQ_OUT_CODES,
                      ifq.IFQ_PATH_DIRECT if in_bits == 8 else ifq.IFQ_PATH_WARP, pool=2, in_bits=in_bits)
    xp = torch.from_numpy(x if in_bits == 8 else synth.pack_codes(x)).cuda()
    prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(d, torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda(), prep)
    y = torch.full((*A.shape[:3], cout // 4), 0x5A, dtype=torch.uint8, device="cuda")
    ifq.ifq_conv2bit(d, xp, prep, torch.from_numpy(T).cuda(), torch.from_numpy(s).cuda(), y, None)
    assert ifq.ifq_device_status() == ifq.IFQ_OK
    assert (synth.unpack_codes(y.cpu().numpy(), cout) == O.int_chain(A, T, s)).all()
