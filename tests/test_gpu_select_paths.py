"""The top-m selection's kernels by unit length and number of units (a warp per unit up to 256
candidates, up to 512 with more than 4 units per SM and up to 1024 with more than 6; else CTAs of 256, 512 and 1024
threads), bit for bit against the oracle on scores that stress the radix digits: ties,
equal scores, neighbours one ulp apart, all magnitudes and signs, infinities."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_04771_gb300 import reco

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_04771_gb300 import build
    build.build()
    reco.lib()


def _patterns(rng, n):
    one = np.float32(0.37)
    return [
        np.exp(rng.standard_normal(n)).astype(np.float32),
        rng.integers(0, 4, n).astype(np.float32),
        np.full(n, 0.25, np.float32),
        (np.full(n, one).view(np.int32) + rng.integers(0, 5, n).astype(np.int32)).view(np.float32),  # a few ulps
        (rng.standard_normal(n) * 10.0 ** rng.integers(-30, 30, n)).astype(np.float32),
        np.where(rng.random(n) < 0.3, np.float32(-np.inf), np.where(rng.random(n) < 0.3, np.float32(np.inf),
                                                                   np.float32(0.0))).astype(np.float32),
        np.where(rng.random(n) < 0.5, np.float32(1e-45), np.float32(0.0)).astype(np.float32),  # (no -0: sums of probabilities)
        (2.0 ** rng.integers(-126, 127, n)).astype(np.float32),
    ]


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


# B sequences of two units each: a number, or (m, o) for m units per SM and o sequences more (the rules
# have their lines at 1, 2, 3, 4 and 6 units per SM)
@pytest.mark.parametrize("B,most", [(16, m) for m in (1, 5, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 3000, 9001)]
                         + [(B, m) for B in ((1, 0), (1, 1), (2, 0), (2, 1)) for m in (257, 1024, 1025)]
                         + [(B, m) for B in ((3, 0), (3, 1), (4, 0), (4, 1), (6, 0), (6, 1)) for m in (257, 512, 513, 1024)]
                         + [((4, 1), 1025), ((2, 0), 16384), ((2, 0), 16385), (16, 40000)]
                         # eight keys per thread and one more, with 1024, 512 and 256 threads
                         + [(16, 8192), (16, 8193), ((3, 0), 4096), ((3, 0), 4097), ((6, 0), 2048), ((6, 0), 2049)])
def test_selection_by_length(B, most):
    if isinstance(B, tuple):
        B = B[0] * _sms() // 2 + B[1]
    rng = np.random.default_rng(most + 10007 * (B - 16))
    w = 5
    L_cap = most + w
    H = 2
    lens = np.zeros((1, B, H), np.int32)
    keep = np.zeros(B, np.int32)
    scores = np.zeros((1, B, H, L_cap), np.float32)
    for b in range(B):
        L = L_cap if b < 8 else int(rng.integers(w, L_cap + 1))
        lens[0, b] = L
        keep[b] = {0: w, 1: L, 2: min(L, w + 1)}.get(b % 8, int(rng.integers(w, L + 1)))
        for h in range(H):
            scores[0, b, h] = _patterns(rng, L_cap)[(b + h) % 8]
    K = torch.zeros((1, B, H, L_cap, 64), dtype=torch.bfloat16, device=DEV)
    kv = reco.make_kv(K, K.clone(), H)
    kept = torch.full((1, B, H, L_cap), -1, dtype=torch.int32, device=DEV)
    ws = reco.workspace(reco.RECO_OP_SELECT, kv, w, DEV)
    lens_t, keep_t = torch.from_numpy(lens).to(DEV), torch.from_numpy(keep).to(DEV)
    reco.reco_select_topm(kv, torch.from_numpy(scores).to(DEV), lens_t, keep_t, w, kept, ws)
    reco.reco_check()
    got = kept.cpu().numpy()
    for b in range(B):
        for h in range(H):
            L, m = int(lens[0, b, h]), int(keep[b])
            ref = oracle.select_unit(scores[0, b, h, :L], L, w, m)
            np.testing.assert_array_equal(got[0, b, h, :m], ref[:m], err_msg=f"{(b, h, L, m)}")
            if m < L:
                assert (got[0, b, h, m:] == -1).all()
