"""The im2col tensor-core kernel on layers with an odd number of K stages per tile.

Its two MMA warps share the ring of K stages.  Pairs of stages counted from each tile's first stage moved
over the ring's slots when a tile had an odd number of them, and a warp that reached a slot before the
gather had filled the slot's previous stage (the other warp's) went on with stale data: a timeout or a
fault, rarely, on layers of many tiles whose gather is slow (1-byte granules).  Pairs are ring slots now.
"""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1911_08076_gb300 import ifq, synth

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("shape", [(24, 29, 66, 440, 88, 3), (40, 28, 28, 64, 64, 3), (9, 37, 45, 36, 100, 3)],
                         ids=["31stages_1byte", "5stages_16byte", "3stages_1byte"])
def test_odd_stage_counts_over_many_tiles(monkeypatch, shape):
    monkeypatch.setenv("IFQ_BAND", "0")
    n, h, w, cin, cout, k = shape
    rng = np.random.default_rng(5)
    x = rng.integers(0, 4, (n, h, w, cin), dtype=np.uint8)
    wt = np.where(rng.integers(0, 2, (cout, k, k, cin)) == 1, 1, -1).astype(np.int8)
    d = ifq.conv_desc(n, h, w, cin, cout, k, 1, k // 2, ifq.IFQ_OUT_ACC, ifq.IFQ_PATH_TC)
    xp = torch.from_numpy(synth.pack_codes(x)).cuda()
    bits = torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda()
    prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(d, bits, prep)
    first = None
    for _ in range(20):
        y = torch.full((n, h, w, cout), -7, dtype=torch.int32, device="cuda")
        ifq.ifq_conv2bit(d, xp, prep, None, None, None, y)
        assert ifq.ifq_device_status() == ifq.IFQ_OK
        if first is None:
            first = y
            assert (y[:1].cpu().numpy() == O.conv_acc(x[:1], wt, 1, k // 2)).all()
        else:
            assert torch.equal(y, first)
