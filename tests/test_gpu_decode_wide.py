"""Decode with more than 8 query heads per KV head in the kernel that chooses between one pass over
all heads and two halves from the lengths, and units cut into few pieces when they are few: sampled
units against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import DECODE_ATOL, gpu_decode, np32
from paper_2608_04771_gb300 import reco
from paper_2608_04771_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_04771_gb300 import build
    build.build()
    reco.lib()


def _check(wl, lens_np, units):
    g = torch.Generator(device=DEV)
    g.manual_seed(7)
    shape = (wl.layers, wl.batch, wl.h_kv, wl.L_cap, wl.d)
    K = torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)
    V = torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)
    lens = torch.from_numpy(lens_np).to(DEV)
    q, kn, vn = W.make_decode_step(wl, 0, DEV)
    out, lse = gpu_decode(wl, K, V, lens, q, kn, vn)
    reco.reco_check()
    np.testing.assert_array_equal(lens.cpu().numpy(), lens_np + 1)
    for l, b, h in units:
        L = int(lens_np[l, b, h])
        k = np.concatenate([np32(K[l, b, h, :L]), np32(kn[l, b, h:h + 1])])
        v = np.concatenate([np32(V[l, b, h, :L]), np32(vn[l, b, h:h + 1])])
        assert torch.equal(K[l, b, h, L], kn[l, b, h]) and torch.equal(V[l, b, h, L], vn[l, b, h])
        for hq in range(h * wl.G, (h + 1) * wl.G):
            o, z = oracle.decode_unit(np32(q[l, b, hq]), k, v, L + 1, wl.scale())
            assert np.abs(out[l, b, hq].cpu().numpy() - o).max() <= DECODE_ATOL["bf16"], (l, b, hq)
            assert abs(float(lse[l, b, hq]) - z) < 1e-3


# 32 units with room for 16000 rows: halves below 16 blocks a warp (short: whole units; medium: cut),
# one pass above
@pytest.mark.parametrize("G,d", [(9, 64), (13, 128), (16, 128)])
@pytest.mark.parametrize("lo,hi", [(1, 250), (1, 3000), (11000, 15990)])
def test_one_pass_or_halves(G, d, lo, hi):
    wl = W.WORKLOADS["7b"].reduced(layers=4, batch=4, h_q=2 * G, h_kv=2, d=d, L=15999, decode_steps=1)
    lens = np.random.default_rng(G + hi).integers(lo, hi + 1, (4, 4, 2)).astype(np.int32)
    _check(wl, lens, [(0, 0, 0), (1, 3, 1), (3, 3, 1)])


@pytest.mark.parametrize("units,G,L", [(1, 8, 30000), (2, 16, 20000), (6, 5, 5000), (16, 7, 3000)])
def test_few_units(units, G, L):
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=units, h_q=G, h_kv=1, L=L, decode_steps=1)
    lens = np.random.default_rng(L).integers(L // 2, L + 1, (1, units, 1)).astype(np.int32)
    _check(wl, lens, [(0, 0, 0), (0, units - 1, 0)])


# a long unit among short ones: it is cut into as many pieces as balance its merge, whatever the
# number of short units (never cut) beside it
@pytest.mark.parametrize("short,G,L", [(1, 7, 20000), (40, 4, 32000), (600, 7, 32000), (63, 16, 9000)])
def test_one_long_unit_among_short_ones(short, G, L):
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=short + 1, h_q=G, h_kv=1, L=L, decode_steps=1)
    lens = np.random.default_rng(L).integers(1, 250, (1, short + 1, 1)).astype(np.int32)
    long = short // 2
    lens[0, long, 0] = L
    _check(wl, lens, [(0, 0, 0), (0, long, 0), (0, short, 0)])


# units of one length: whole numbers of pieces, also where the cap or the blocks per warp leave a remainder
@pytest.mark.parametrize("units,G,L", [(8, 7, 500), (7, 1, 763), (31, 4, 1500), (3, 16, 9000), (150, 8, 763)])
def test_units_of_one_length(units, G, L):
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=units, h_q=G, h_kv=1, L=L, decode_steps=1)
    _check(wl, np.full((1, units, 1), L - 1, np.int32), [(0, 0, 0), (0, units // 2, 0), (0, units - 1, 0)])


def test_no_unit_with_keys():
    wl = W.WORKLOADS["7b"].reduced(layers=1, batch=3, h_q=2, h_kv=1, L=64, decode_steps=1)
    K, V = W.make_cache(wl, DEV, canary=False)
    q, _, _ = W.make_decode_step(wl, 0, DEV)
    out, lse = gpu_decode(wl, K, V, torch.zeros((1, 3, 1), dtype=torch.int32, device=DEV), q)
    reco.reco_check()
    assert torch.all(out == 0) and torch.all(torch.isneginf(lse))
