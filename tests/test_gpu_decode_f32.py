"""Decode attention over float32 caches on the streamed kernel, against the oracle: every head
count's register layout (2, 4 and 8 heads, halves above 8), both head dimensions, lengths around a
block of 8 keys, units cut between warps and merged, more units than one launch plans, the rings."""
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


def _wl(G, h_kv, d, L, layers=1, batch=1, steps=2):
    return W.WORKLOADS["tiny"].reduced(layers=layers, batch=batch, h_q=G * h_kv, h_kv=h_kv, d=d, L=L, decode_steps=steps)


def _check(wl, lens_np, append, units=None, out_dtype=torch.float32, step=0):
    K, V = W.make_cache(wl, DEV, canary=False)
    lens = torch.from_numpy(lens_np).to(DEV)
    rows = torch.arange(wl.L_cap, device=DEV)
    past = rows.view(1, 1, 1, -1) >= lens.unsqueeze(-1)
    K.masked_fill_(past.unsqueeze(-1), float("nan"))  # rows past the lengths are never read
    V.masked_fill_(past.unsqueeze(-1), float("nan"))
    q, kn, vn = W.make_decode_step(wl, step, DEV)
    out, lse = gpu_decode(wl, K, V, lens, q, kn if append else None, vn if append else None, out_dtype)
    reco.reco_check()
    G = wl.G
    units = list(np.ndindex(*lens_np.shape)) if units is None else units
    for l, b, h in units:
        L = int(lens_np[l, b, h])
        k, v = np32(K[l, b, h, :L]), np32(V[l, b, h, :L])
        if append:
            k, v = np.concatenate([k, np32(kn[l, b, h:h + 1])]), np.concatenate([v, np32(vn[l, b, h:h + 1])])
            np.testing.assert_array_equal(np32(K[l, b, h, L]), np32(kn[l, b, h]))  # the new row landed
            np.testing.assert_array_equal(np32(V[l, b, h, L]), np32(vn[l, b, h]))
            assert int(lens[l, b, h]) == L + 1
        for g in range(h * G, (h + 1) * G):
            o, z = oracle.decode_unit(np32(q[l, b, g]), k, v, k.shape[0], wl.scale())
            got = out[l, b, g].float().cpu().numpy()
            tol = DECODE_ATOL["f32"] + (np.abs(o) * 2.0 ** -8 if out_dtype == torch.bfloat16 else 0.0)
            assert (np.abs(got - o) <= tol).all(), (l, b, g, np.abs(got - o).max())
            assert abs(float(lse[l, b, g]) - z) < 1e-4


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("append", [False, True])
def test_head_counts_and_block_edges(G, d, append):
    wl = _wl(G, 5, d, 400, batch=2)
    lens = np.array([[[1, 7, 8, 9, 400], [128, 129, 136, 250, 15]]], np.int32)
    _check(wl, lens, append)


@pytest.mark.parametrize("G,L", [(6, 40000), (16, 9000)])
def test_units_cut_between_warps(G, L):
    _check(_wl(G, 2, 128, L), np.array([[[L, L // 2 + 3]]], np.int32), True, out_dtype=torch.bfloat16)


def test_first_appended_row_and_no_room():
    wl = _wl(6, 2, 128, 16, steps=0)
    K, V = W.make_cache(wl, DEV, canary=False)
    q, kn, vn = W.make_decode_step(wl.reduced(decode_steps=1), 0, DEV)
    lens = torch.tensor([[[0, 16]]], dtype=torch.int32, device=DEV)  # an empty unit; a full one
    out, lse = gpu_decode(wl, K, V, lens, q, kn, vn)
    with pytest.raises(reco.RecoError) as e:
        reco.reco_check()
    assert e.value.status == reco.RECO_EDEVICE
    # one key: its value row, with probability one
    assert torch.equal(out[0, 0, :6], vn[0, 0, 0].expand(6, -1))
    assert torch.all(out[0, 0, 6:] == 0) and torch.all(torch.isneginf(lse[0, 0, 6:]))
    assert lens.tolist() == [[[1, 16]]]
    reco.reco_check()


@pytest.mark.parametrize("G", [2, 9])  # parts of 7168 units, of 3584 with two halves per unit
def test_more_units_than_one_launch(G):
    wl = _wl(G, 8, 64, 40, layers=10, batch=91)
    lens = np.random.default_rng(G).integers(0, 41, (10, 91, 8)).astype(np.int32)
    rng = np.random.default_rng(1)
    units = [tuple(int(x) for x in np.unravel_index(i, lens.shape)) for i in rng.integers(0, lens.size, 60)]
    _check(wl, lens, True, [u for u in units + [(9, 90, 7), (0, 0, 0)]])


def test_rings():
    wl = _wl(9, 2, 128, 300, batch=2)
    K, V = W.make_cache(wl, DEV, canary=False)
    lens = torch.full((1, 2, 2), 290, dtype=torch.int32, device=DEV)
    S, n = 3, 2 * wl.h_q
    ring = torch.zeros((2 * S, n), dtype=torch.float32, device=DEV)
    q_ring = torch.zeros((1, 2, wl.h_q, S, 128), dtype=torch.float32, device=DEV)
    slot = torch.tensor([1], dtype=torch.long, device=DEV)
    kv = reco.make_kv(K, V, wl.h_q)
    ws = reco.workspace(reco.RECO_OP_DECODE, kv, 0, DEV)
    for t in range(4):
        q, kn, vn = W.make_decode_step(wl, t, DEV)
        ref_l = lens.clone()
        ref_o, ref_lse = gpu_decode(wl, K.clone(), V.clone(), ref_l, q, kn, vn)
        out = torch.empty_like(ref_o)
        s = int(slot)
        reco.reco_decode_attn_ring(kv, q, kn, vn, lens, wl.scale(), out, ring, slot, ws, q_ring=q_ring)
        reco.reco_check()
        assert torch.equal(out, ref_o) and torch.equal(lens, ref_l)
        assert torch.equal(ring[s], ref_lse.flatten()) and torch.equal(ring[s + S], ref_lse.flatten())
        assert torch.equal(q_ring[..., s, :], q) and int(slot) == (s + 1) % S


def test_rounding_does_not_grow_with_the_keys():
    """Errors against float64. An output is a sum of about n = 720 random terms in one warp: added one by one,
    each rounding (2^-24 / sqrt(3) of the partial sum on average over its binade) would give
    1.7e-8 * sqrt(n / 2) = 3.2e-7 of the result, blocks of 8 first 1.1e-7; the exponentials and logits add
    about 2e-7 in either case."""
    wl = _wl(8, 4, 128, 1155, layers=12, batch=21, steps=1)
    lens_np = np.random.default_rng(5).integers(577, 1156, (12, 21, 4)).astype(np.int32)
    K, V = W.make_cache(wl, DEV, canary=False)
    q, _, _ = W.make_decode_step(wl, 0, DEV)
    out, _ = gpu_decode(wl, K, V, torch.from_numpy(lens_np).to(DEV), q)
    reco.reco_check()
    num = den = 0.0
    for l, b, h in [(l, b, h) for l in range(0, 12, 3) for b in range(0, 21, 5) for h in range(4)]:
        n, hq = int(lens_np[l, b, h]), slice(8 * h, 8 * h + 8)
        p = torch.softmax(q[l, b, hq].double() @ K[l, b, h, :n].double().T * wl.scale(), 1)
        ref = p @ V[l, b, h, :n].double()
        num += float((out[l, b, hq].double() - ref).square().sum())
        den += float(ref.square().sum())
    assert (num / den) ** 0.5 < 3e-7
