"""The band kernel (4-bit products on an input band expanded once) on every launch shape of its table, bit-exact
against the CPU oracle: ragged maps and channel tiles, each load granule (16, 8, 4, 2 and 1 bytes), odd plane
counts, several chunks and tiles, strided 1 x 1 filters, 2-, 3- and 4-bit codes, and thresholds that saturate or are not
equally spaced (one comparison after the fitted line, or a search).  The results are integers: no tolerance."""
import re

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1911_08076_gb300 import ifq, synth

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# Launch shapes, as IFQ_BAND asks for them: 64 channels a tile, the same and two channel tiles a CTA, the same and two
# subtiles; 128 channels, .. two tiles, .. two subtiles with streamed filters.
SHAPES = (2, 3, 4, 5, 6, 7)
CASES = [
    # n, h, w, cin, cout, k, stride, pad, bits per code, the shapes that fit (two channel tiles need that many channels,
    # resident filters their shared memory)
    (2, 16, 16, 64, 64, 3, 1, 1, 2, (2, 4, 5, 7)),            # 16-byte granules, one tile of channels
    (3, 11, 13, 128, 256, 3, 1, 1, 2, SHAPES),                # several tiles with ragged tails
    (9, 37, 45, 72, 100, 3, 1, 1, 2, (2, 3, 4, 5, 7)),        # 2-byte granules, an odd plane, ragged channels
    (2, 9, 9, 36, 132, 3, 1, 2, 2, SHAPES),                   # 1-byte granules, two channel tiles, the last one ragged
    (2, 8, 9, 32, 40, 3, 1, 1, 2, (2, 4, 5, 7)),              # one plane: taps in pairs, the last alone
    (2, 12, 12, 16, 36, 3, 1, 1, 2, (2, 4, 5, 7)),            # 4-byte granules
    (1, 27, 27, 96, 64, 5, 1, 2, 2, (2, 4, 5, 7)),            # 25 taps, 8-byte granules
    (4, 7, 7, 512, 192, 3, 1, 1, 2, (2, 4, 7)),               # 16 planes in chunks
    (2, 8, 8, 256, 320, 1, 1, 0, 2, SHAPES),                  # 1 x 1 on the map as it lies
    (3, 15, 14, 64, 72, 1, 2, 0, 2, (2, 3, 4, 5, 7)),         # strided 1 x 1
    (40, 13, 13, 32, 64, 3, 1, 0, 2, (2, 4, 5, 7)),           # no padding, 53 tiles
    (2, 9, 9, 24, 40, 3, 1, 1, 4, (2, 4, 5, 7)),
    (3, 14, 10, 40, 96, 3, 1, 1, 3, (2, 3, 4, 5, 7)),
    (2, 13, 13, 384, 136, 3, 1, 1, 4, (7,)),                  # 24 planes of digits
]


def _thresholds(rng, cout, K, kbits, spacing):
    """Ascending thresholds across the accumulator's spread: floors of equally spaced values ("even"), some of them a
    fraction of a step off ("near", as the separated conversion's), or any ("far").  By the kernel's fit a line is the
    code, the code or one below it, or neither; the last two only in some columns of a block."""
    L = (1 << kbits) - 1
    sd = np.sqrt(K * L * (2 * L + 1) / 6.0)
    step, base = rng.uniform(0.3, 1.0, cout) * 3 * sd / L, rng.normal(0, 0.3 * sd, cout)
    step[1::5] *= 10.0 ** rng.integers(-1, 5, step[1::5].shape)   # steep ones, and thresholds past the bound L K
    T = np.floor(base[:, None] + step[:, None] * (np.arange(L) - (L - 1) / 2))
    if spacing == "near":
        T[::4] += np.floor(rng.uniform(-0.2, 0.2, T[::4].shape) * step[::4, None])
        T.sort(axis=1)
    elif spacing == "far":
        T[::3] += np.cumsum(rng.integers(0, int(sd) + 2, T[::3].shape), axis=1)
    return np.clip(T, -L * K - 1, L * K).astype(np.int32), np.where(rng.integers(0, 4, cout) == 0, -1, 1).astype(np.int8)


@pytest.mark.parametrize("case", CASES, ids=[f"c{c[3]}x{c[4]}k{c[5]}s{c[6]}b{c[8]}" for c in CASES])
def test_every_launch_shape_matches_oracle(case, monkeypatch):
    n, h, w, cin, cout, k, stride, pad, kbits, shapes = case
    rng = np.random.default_rng(cin * 131 + cout)
    x = rng.integers(0, 1 << kbits, (n, h, w, cin), dtype=np.uint8)
    wt = np.where(rng.integers(0, 2, (cout, k, k, cin)) == 1, 1, -1).astype(np.int8)
    A = O.conv_acc(x, wt, stride, pad)
    d = ifq.conv_desc(n, h, w, cin, cout, k, stride, pad, ifq.IFQ_OUT_BOTH, ifq.IFQ_PATH_TC, kbits=kbits)
    xp = torch.from_numpy(synth.pack_codes(x, kbits)).cuda()
    prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(d, torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda(), prep)
    rowb = cout * synth.field_bits(kbits) // 8
    for spacing in ("even", "near", "far"):
        T, s = _thresholds(rng, cout, k * k * cin, kbits, spacing)
        C = O.int_chain(A, T, s)
        for shape in (1, *shapes):   # 1: the planner's choice
            monkeypatch.setenv("IFQ_BAND", str(shape))
            assert shape == 1 or ifq.ifq_conv_kernel(d).startswith("conv_band_kernel")
            yc = torch.full((*A.shape[:3], rowb), 0x5A, dtype=torch.uint8, device="cuda")
            ya = torch.full(A.shape, -777777, dtype=torch.int32, device="cuda")
            ifq.ifq_conv2bit(d, xp, prep, torch.from_numpy(T).cuda(), torch.from_numpy(s).cuda(), yc, ya)
            assert ifq.ifq_device_status() == ifq.IFQ_OK
            assert (ya.cpu().numpy() == A).all(), shape
            assert (synth.unpack_codes(yc.cpu().numpy(), cout, kbits) == C).all(), (shape, spacing)


MANY = [
    # cin, cout, k, bits per code: every launch shape, several rounds of every ring in each CTA
    (32, 200, 3, 2),      # 8-byte granules, one plane
    (68, 136, 3, 2),      # 1-byte granules, three planes
    (64, 132, 3, 2),      # 16-byte granules
    (8, 136, 5, 2),       # 2-byte granules, 25 taps
    (288, 136, 1, 2),     # three chunks a tile
    (256, 200, 1, 2),     # 1 x 1: the epilogue sets the pace
    (40, 200, 3, 3),      # 4-byte granules
    (24, 136, 3, 4),      # two tiles of 128 channels a CTA: the fit's table is full
    (128, 256, 1, 4),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("case", MANY, ids=[f"c{c[0]}x{c[1]}k{c[2]}b{c[3]}" for c in MANY])
def test_many_tiles_per_cta(case, shape, monkeypatch):
    """Persistent CTAs that go round their accumulators, barrier pairs, chunk and filter rings several times, by lines and by
    comparisons, three runs of each.  The reference is float64 torch."""
    cin, cout, k, kbits = case
    n, h, w, pad, top = 620, 13, 13, k // 2, (1 << kbits) - 1
    monkeypatch.setenv("IFQ_BAND", str(shape))
    d = ifq.conv_desc(n, h, w, cin, cout, k, 1, pad, ifq.IFQ_OUT_BOTH, ifq.IFQ_PATH_TC, kbits=kbits)
    plan = dict(re.findall(r"(\w+)=(\d+)", ifq.ifq_conv_kernel(d)))
    assert int(plan["units"]) > 2 * int(plan["accumulators"])
    rng = np.random.default_rng(cin + 7 * cout)
    x = rng.integers(0, top + 1, (n, h, w, cin), dtype=np.uint8)
    wt = np.where(rng.integers(0, 2, (cout, k, k, cin)) == 1, 1, -1).astype(np.int8)
    xd = torch.nn.functional.pad(torch.from_numpy(x).cuda().double(), (0, 0, pad, pad, pad, pad))
    wd = torch.from_numpy(wt).cuda().double()
    A = sum(xd[:, i:i + h, j:j + w] @ wd[:, i, j].T for i in range(k) for j in range(k))
    prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(d, torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda(), prep)
    xp = torch.from_numpy(synth.pack_codes(x, kbits)).cuda()
    for spacing in ("even", "near", "far"):
        T, s = _thresholds(rng, cout, k * k * cin, kbits, spacing)
        td, sd = torch.from_numpy(T).cuda(), torch.from_numpy(s).cuda()
        C = sum((A * sd > td[:, i]).to(torch.uint8) for i in range(top))
        for _ in range(3):
            yc = torch.full((n, h, w, cout * synth.field_bits(kbits) // 8), 0x5A, dtype=torch.uint8, device="cuda")
            ya = torch.full((n, h, w, cout), -777777, dtype=torch.int32, device="cuda")
            ifq.ifq_conv2bit(d, xp, prep, td, sd, yc, ya)
            assert ifq.ifq_device_status() == ifq.IFQ_OK
            assert torch.equal(ya.double(), A), spacing
            codes = torch.empty(n * h * w * cout, dtype=torch.uint8, device="cuda")
            ifq.ifq_unpack_codes_kbits(yc, codes, codes.numel(), kbits)
            assert torch.equal(codes.view(C.shape), C), spacing


@pytest.mark.parametrize("kbits,K", [(2, 65536), (3, 28064), (4, 13088)])
def test_accumulation_exact_at_the_admitted_bound(kbits, K, monkeypatch):
    """Accumulators up to the largest magnitude admitted, (2^k - 1) K <= 196608, with small odd addends all along
    K: the 4-bit products' fp32 sums must stay exact.  The sums are checked against float64.  Filters of that K
    are streamed (one launch shape); the products and sums are the same instructions in every shape."""
    rng = np.random.default_rng(K)
    L = (1 << kbits) - 1
    n, cout = 300, 72
    x = rng.choice(np.array([1, 2, L - 1, L], np.uint8), size=(n, 1, 1, K), p=[0.05, 0.05, 0.1, 0.8])
    x[0] = L
    wt = np.ones((cout, 1, 1, K), np.int8)
    wt[1] = -1
    for r in range(2, cout):
        wt[r, 0, 0, rng.random(K) < (0.05 if r < 40 else 0.5)] = -1
    A = (x.reshape(n, K).astype(np.float64) @ wt.reshape(cout, K).astype(np.float64).T).astype(np.int64)
    d = ifq.conv_desc(n, 1, 1, K, cout, 1, 1, 0, ifq.IFQ_OUT_ACC, ifq.IFQ_PATH_TC, kbits=kbits)
    xp = torch.from_numpy(synth.pack_codes(x, kbits)).cuda()
    prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(d, torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda(), prep)
    for shape in (7,):
        monkeypatch.setenv("IFQ_BAND", str(shape))
        assert ifq.ifq_conv_kernel(d).startswith("conv_band_kernel")
        ya = torch.full((n, 1, 1, cout), -777777, dtype=torch.int32, device="cuda")
        ifq.ifq_conv2bit(d, xp, prep, None, None, None, ya)
        assert ifq.ifq_device_status() == ifq.IFQ_OK
        assert (ya.cpu().numpy().reshape(n, cout) == A).all(), shape


@pytest.mark.parametrize("kbits", [2, 4])
@pytest.mark.parametrize("prepared", ["pooled", "strided", "fully connected", "bit-serial"])
def test_filters_prepared_for_another_layer_with_them(prepared, kbits, monkeypatch):
    """Filters prepared from a descriptor that the band kernel does not serve run on it from one that it does."""
    n, h, w, cin, cout, k = 3, 12, 14, 64, 72, 3
    rng = np.random.default_rng(7)
    x = rng.integers(0, 1 << kbits, (n, h, w, cin), dtype=np.uint8)
    wt = np.where(rng.integers(0, 2, (cout, k, k, cin)) == 1, 1, -1).astype(np.int8)
    dp = {"pooled": ifq.conv_desc(1, h, w, cin, cout, k, 1, 1, pool=2, kbits=kbits),
          "strided": ifq.conv_desc(1, h, w, cin, cout, k, 2, 1, kbits=kbits),
          "fully connected": ifq.conv_desc(1, k, k, cin, cout, k, 1, 0, kbits=kbits),
          "bit-serial": ifq.conv_desc(1, h, w, cin, cout, k, 3, 1, path=ifq.IFQ_PATH_BITSERIAL, kbits=kbits)}[prepared]
    d = ifq.conv_desc(n, h, w, cin, cout, k, 1, 1, ifq.IFQ_OUT_ACC, ifq.IFQ_PATH_TC, kbits=kbits)
    assert ifq.ifq_weights_prep_bytes(dp) == ifq.ifq_weights_prep_bytes(d)
    prep = torch.empty(ifq.ifq_weights_prep_bytes(dp), dtype=torch.uint8, device="cuda")
    ifq.ifq_pack_weights(dp, torch.from_numpy(synth.pack_signs(wt).view(np.int32)).cuda(), prep)
    monkeypatch.setenv("IFQ_BAND", "2")
    ya = torch.full((n, h, w, cout), -777777, dtype=torch.int32, device="cuda")
    ifq.ifq_conv2bit(d, torch.from_numpy(synth.pack_codes(x, kbits)).cuda(), prep, None, None, None, ya)
    assert ifq.ifq_device_status() == ifq.IFQ_OK
    assert (ya.cpu().numpy() == O.conv_acc(x, wt, 1, 1)).all()
