"""The tensor-core scoring's work plan and column ranges, and the pool's tiles, against the oracle:
window-row counts whose halves end in 8 columns, ranges of more than one plan round, pools that
cross tiles, exceed the shared-memory halo or meet unaligned rows."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_scores_close, gpu_score, np32
from paper_2608_04771_gb300 import reco
from paper_2608_04771_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_04771_gb300 import build
    build.build()
    reco.lib()


def _check(wl, lens, pool, units):
    K, V = W.make_cache(wl, DEV, canary=False)
    q = W.make_qwin(wl, DEV)
    got = gpu_score(wl, K, V, q, torch.from_numpy(lens).to(DEV), pool).cpu().numpy()
    reco.reco_check()
    G = wl.h_q // wl.h_kv
    for l, b, h in units:
        L = int(lens[l, b, h])
        _, ora = oracle.score_unit(np32(q[l, b, h * G:(h + 1) * G]), np32(K[l, b, h, :L]), wl.w, wl.scale(), pool)
        assert_scores_close(got[l, b, h, :L - wl.w], ora, f"unit {(l, b, h)}")


# window rows G * w: 5 and 16 (one 8-column half), 48 (16 + 8), 112, 130 (144 columns, three regions),
# 272 (two chains of 144), 384 (three query tiles), 400 and 512 (four)
@pytest.mark.parametrize("G,w,d", [(1, 5, 64), (1, 16, 128), (3, 16, 128), (7, 16, 64), (13, 10, 128), (17, 16, 128),
                                   (12, 32, 64), (8, 50, 128), (16, 32, 128)])
def test_window_row_counts(G, w, d):
    wl = W.WORKLOADS["7b"].reduced(layers=2, batch=2, h_q=2 * G, h_kv=2, d=d, L=2300, decode_steps=5, w=w)
    rng = np.random.default_rng(G * 100 + w)
    lens = rng.integers(w, 2306, (2, 2, 2)).astype(np.int32)
    lens[0, 0, 0], lens[1, 1, 1] = 2048 + w, w + 1
    _check(wl, lens, 7, [(0, 0, 0), (0, 1, 1), (1, 0, 0), (1, 1, 1)])


def test_more_units_than_one_plan_round():
    """About 300 units per CTA of one or two tiles each: two rounds of 256 runs."""
    wl = W.WORKLOADS["7b"].reduced(layers=64, batch=89, h_q=8, h_kv=8, d=64, L=200, decode_steps=0, w=8)
    rng = np.random.default_rng(3)
    lens = rng.integers(8, 201, (64, 89, 8)).astype(np.int32)
    units = [tuple(int(x) for x in np.unravel_index(i, lens.shape)) for i in rng.integers(0, lens.size, 40)]
    _check(wl, lens, 3, units + [(0, 0, 0), (63, 88, 7)])


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("L,pool", [(4240, 7), (4241, 9), (4240, 21), (4243, 129), (4240, 131), (8300, 1)])
def test_pool_tiles(dtype, L, pool):
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=1, h_q=4, h_kv=2, d=64, L=L, decode_steps=0, w=16, dtype=dtype)
    _check(wl, np.array([[[L, 4096 + 17 if L < 8000 else 4111]]], np.int32), pool, [(0, 0, 0), (0, 0, 1)])


# plain-FMA passes: rows below, at and past a 64-row tile, units shorter than one key tile, ragged
@pytest.mark.parametrize("G,w,d", [(1, 5, 64), (4, 16, 128), (13, 5, 128), (6, 32, 128), (10, 39, 128), (12, 64, 64)])
def test_f32_row_counts(G, w, d):
    wl = W.WORKLOADS["7b"].reduced(layers=2, batch=2, h_q=2 * G, h_kv=2, d=d, L=1500, decode_steps=5, w=w, dtype="f32")
    rng = np.random.default_rng(G * 100 + w)
    lens = rng.integers(w, 1506, (2, 2, 2)).astype(np.int32)
    lens[0, 0, 0], lens[0, 1, 1], lens[1, 1, 1] = 1505, 128 + w, w + 1
    _check(wl, lens, 7, [(0, 0, 0), (0, 1, 1), (1, 0, 0), (1, 1, 1)])


def test_bf16_rows_beyond_the_tensor_cores():
    """R = 760 window rows at d = 64: the plain-FMA passes read bf16 rows."""
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=2, h_q=38, h_kv=2, d=64, L=700, decode_steps=0, w=40)
    _check(wl, np.array([[[700, 333], [40, 168]]], np.int32), 7, [(0, 0, 0), (0, 0, 1), (0, 1, 1)])


@pytest.mark.parametrize("dtype,G,w,one_pass", [("f32", 1, 5, False), ("f32", 3, 32, False), ("f32", 3, 32, True),
                                                ("f32", 2, 32, True), ("bf16", 19, 40, False)])
def test_minus_infinity_in_a_key(dtype, G, w, one_pass):
    """A key whose logit is -inf in every window row gets score 0 and changes no other score, also where
    the rows end inside a 64-row tile: the same scores as with a finite element that underflows."""
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=1, h_q=2 * G, h_kv=2, d=64, L=300, decode_steps=0, w=w, dtype=dtype)
    K, V = W.make_cache(wl, DEV, canary=False)
    q = W.make_qwin(wl, DEV)
    q[..., 0] = q[..., 0].abs() + 0.5
    lens = torch.full((1, 1, 2), 300, dtype=torch.int32, device=DEV)
    lse = torch.full((w, 1, 1, 2 * G), 6.0, dtype=torch.float32, device=DEV)
    got = []
    for x in (-float("inf"), -1e30):
        K[0, 0, :, 20, 0] = x
        if one_pass:
            kv = reco.make_kv(K, V, wl.h_q)
            scores = torch.zeros(K.shape[:4], dtype=torch.float32, device=DEV)
            ws = reco.workspace(reco.RECO_OP_SCORE, kv, w, DEV)
            reco.reco_score_cache_lse(kv, q, lens, lse, w, 1, wl.scale(), scores, ws)
        else:
            scores = gpu_score(wl, K, V, q, lens, 1)
        reco.reco_check()
        got.append(scores)
    assert torch.all(got[0][0, 0, :, 20] == 0)
    assert torch.equal(got[0], got[1])


# short units: a CTA per item (few units), a planned call whose threads hold 1 to 4 units' lengths, more
# units than that; one and two query tiles of split columns, three and two chains of whole tiles
@pytest.mark.parametrize("layers,G,w,d,L", [(1, 4, 32, 128, 250), (1, 7, 32, 64, 1020), (2, 3, 16, 128, 120), (1, 10, 32, 128, 500),
                                            (30, 8, 32, 128, 300), (160, 1, 5, 64, 140), (300, 2, 8, 64, 130),
                                            (600, 1, 5, 64, 140), (30, 9, 32, 128, 200), (30, 5, 64, 128, 200)])
def test_short_units(layers, G, w, d, L):
    wl = W.WORKLOADS["7b"].reduced(layers=layers, batch=2, h_q=2 * G, h_kv=2, d=d, L=L, decode_steps=4, w=w)
    rng = np.random.default_rng(layers + L)
    lens = rng.integers(w, L + 1, (layers, 2, 2)).astype(np.int32)
    lens[0, 0, 0], lens[0, 1, 1], lens[-1, 1, 0] = w, w + 1, L
    units = [(0, 0, 0), (0, 1, 1), (layers - 1, 1, 0)] + [(int(rng.integers(layers)), b, h) for b in (0, 1) for h in (0, 1)]
    _check(wl, lens, 5, units)
    # one pass with given normalisers, sequence 1 masked out, in float64
    K, V = W.make_cache(wl, DEV, canary=False)
    q = W.make_qwin(wl, DEV)
    kv = reco.make_kv(K, V, wl.h_q)
    scores = torch.full(K.shape[:4], -1.0, dtype=torch.float32, device=DEV)
    lse = torch.linspace(3.0, 6.0, w * layers * 2 * wl.h_q, device=DEV).view(w, layers, 2, wl.h_q)
    keep = torch.tensor([0, 1 << 30], dtype=torch.int32, device=DEV)
    reco.reco_score_cache_lse(kv, q, torch.from_numpy(lens).to(DEV), lse, w, 1, wl.scale(), scores,
                              reco.workspace(reco.RECO_OP_SCORE, kv, w, DEV), keep=keep)
    reco.reco_check()
    assert torch.all(scores[:, 1] == -1.0)
    for l, b, h in units:
        if b == 1:
            continue
        n = int(lens[l, b, h]) - w
        x = torch.einsum("gtd,jd->gtj", q[l, b, h * G:(h + 1) * G].double(), K[l, b, h, :n].double()) * wl.scale()
        ref = torch.exp(x - lse[:, l, b, h * G:(h + 1) * G].double().T.unsqueeze(-1)).sum((0, 1)) / G
        assert_scores_close(scores[l, b, h, :n].cpu().numpy(), ref.cpu().numpy(), f"unit {(l, b, h)}")
