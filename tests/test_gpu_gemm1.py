"""GPU parity of the up-stream stage (gather + grouped GEMM1 + gated activation) against the CPU
oracle, through the C ABI."""

from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import gemm1_act_ref as g1
from oracle import gemm2_combine_ref as g2
from oracle import routing_ref as rr
from paper_2609_07536_b200 import binding as B
from paper_2609_07536_b200 import workloads as wl
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _run(w, idx, hidden, W1, counts_on_device=False):
    h = G.handle()
    ws, idx_d, S = G.build_routing(w, idx, None)
    shape = ws.shape
    hr = torch.empty(B.moe_gemm1_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    x = torch.full((w.R, w.I), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moe_gemm1_act(h, hidden.cuda(), W1.cuda(), shape, w.tile_m, ws.routing,
                    B.MOE_MTILES_ON_DEVICE if counts_on_device else S, hr, x, ws.status)
    torch.cuda.synchronize()
    assert B.moe_get_status(h, ws.status).code == 0
    return x, ws


def _tolerance(ref):
    # bf16 output: its own rounding (2^-9 relative, 2^-8 allowed) on top of the path's tolerance
    rms = float(np.sqrt(np.mean(ref.astype(np.float64) ** 2))) if ref.size else 0.0
    return 1e-2 * rms + 1e-3 + 2.0 ** -8 * np.abs(ref)


def _check(w, n_rows=None, **kw):
    idx, _, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    x, ws = _run(w, idx, hidden, W1, **kw)
    r = rr.build_routing(idx, w.E_tot, w.tile_m)
    if n_rows is None or n_rows >= w.R:
        rows = np.arange(w.R, dtype=np.int32)
    else:
        rng = np.random.default_rng(1)
        pick = set(rng.choice(w.R, size=n_rows, replace=False).tolist())
        for e in range(w.E_tot):                       # first and last row of every expert, rows of partial m-tiles
            lo, hi = int(r["offsets"][e]), int(r["offsets"][e + 1])
            if hi > lo:
                pick.update({lo, hi - 1, lo + (hi - lo - 1) // 128 * 128})
        rows = np.array(sorted(pick), dtype=np.int32)
    ref = g1.gemm1_act(wl.bf16_bits(hidden), wl.bf16_bits(W1), idx, r["perm"], rows=rows)
    got = x.float().cpu().numpy()[rows]
    assert not np.isnan(got).any()
    assert np.all(np.abs(got - ref) <= _tolerance(ref)), float(np.max(np.abs(got - ref)))
    return x, ws, idx, r


def test_tiny_all_rows():
    _check(wl.TINY)


@pytest.mark.parametrize("kw", [
    dict(T=1, E=4, k=2, H=64, I=16, tile_m=64),                       # one token, a 16-column tile
    dict(T=333, E=12, k=3, H=272, I=208, tile_m=64, EP=1),            # ragged rows, partial k-block and n-tile
    dict(T=1030, E=70, k=2, H=512, I=384, tile_m=128),                # empty experts
    dict(T=700, E=6, k=2, n_shared=2, H=256, I=128, tile_m=256, tile_n=256),  # shared experts, 256-row m-tiles
], ids=lambda kw: "-".join(f"{k}{v}" for k, v in kw.items()))
def test_edge_shapes(kw):
    base = dict(name="g1edge", routing_seed=7, data_seed=8, TP=1, EP=1, L=1, tile_n=64)
    base.update(kw)
    _check(replace(wl.TINY, **base))


def test_granite_and_dsv2lite_shapes_sampled():
    _check(wl.GRANITE, n_rows=300)
    _check(wl.DSV2L, n_rows=200, counts_on_device=True)


def test_same_bits_for_every_m_tile_size():
    # the m-tile size only changes which CTA computes a row, never the arithmetic of the row
    w = replace(wl.GRANITE, name="g1bits", T=900)
    idx, _, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    base = None
    for tm in (64, 128, 256):
        x, _ = _run(replace(w, tile_m=tm), idx, hidden, W1)
        bits = x.view(torch.int16).cpu().numpy()
        if base is None:
            base = bits
        assert np.array_equal(base, bits), tm


@pytest.mark.parametrize("H", [64, 128, 272, 448, 2048])      # 1, 2, 5, 7, 32 k-blocks a tile: seven stages
def test_pair_hand_over_repeats_the_same_bits(H):
    # more tiles than pairs, so that the stages wrap inside and across tiles
    w = replace(wl.TINY, name="g1pair", T=1030, E=4, k=2, H=H, I=2048, TP=1, EP=1, L=1, tile_m=128, tile_n=64)
    idx, _, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    base, _ = _run(w, idx, hidden, W1)
    for _ in range(3):
        x, _ = _run(replace(w, tile_m=256, tile_n=256), idx, hidden, W1)
        assert torch.equal(x.view(torch.int16), base.view(torch.int16))


@pytest.mark.parametrize("tile_m", [64, 128, 256])
def test_activation_over_its_whole_range(tile_m):
    # one-hot hidden states and unit up rows make g a stored bf16 number and the product silu(g) itself.  The fp32 value
    # may be off by __expf's documented 2 + floor(1.173 |g|) ulp, half an ulp each for the sum and the quotient, and one for
    # the reference's own rounding; the stored bf16 is then the rounding of a number in that interval.
    T, H, I = 64, 64, 128
    w = replace(wl.TINY, name="g1silu", T=T, E=1, k=1, n_shared=0, H=H, I=I, TP=1, EP=1, L=1, tile_m=tile_m, tile_n=256 if tile_m == 256 else 64)
    exps, mants = np.arange(-22, 10), np.arange(128)          # 2^-22 .. 1020, both signs, all mantissas
    mag = (2.0 ** exps[:, None] * (1.0 + mants[None, :] / 128.0)).ravel()
    g = np.concatenate([mag, -mag])
    assert g.size == T * I
    W1 = torch.ones((1, 2, I, H), dtype=torch.bfloat16)
    W1[0, 0] = torch.from_numpy(g.reshape(T, I).T.copy()).to(torch.bfloat16)
    hidden = torch.eye(T, H, dtype=torch.bfloat16)
    x, _ = _run(w, np.zeros((T, 1), np.int32), hidden, W1)
    got = x.float().cpu().numpy().astype(np.float64).ravel()
    ref = g / (1.0 + np.exp(-np.maximum(g, -700.0)))
    delta = (4.0 + np.floor(1.173 * np.abs(g))) * 2.0 ** -23
    lo, hi = (torch.from_numpy(ref * (1.0 + sgn * delta)).to(torch.float32).to(torch.bfloat16).double().numpy() for sgn in (-1.0, 1.0))
    far = g < -88.0                                           # exp(-g) overflows fp32 there: -0, for results under 1e-36
    assert np.all((got >= np.minimum(lo, hi))[~far]) and np.all((got <= np.maximum(lo, hi))[~far])
    assert np.all(np.abs(got[far]) <= 1e-36)


def test_output_feeds_the_down_projection():
    # GEMM1's x_routed goes straight into GEMM2 + combine; the layer's output matches the oracle's GEMM2
    # evaluated on the very bits GEMM1 produced
    w = replace(wl.TINY, name="chain", T=300, E=6, k=2, H=128, I=128, TP=1, EP=2, tile_m=128, tile_n=128)
    idx, wt, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    _, W2 = wl.make_data(w)
    x, ws = _run(w, idx, hidden, W1)
    outs, plan, ws2, S, st = G.run_layer(w, idx, wt, x, W2, ws=ws)
    assert st.code == 0
    r = rr.build_routing(idx, w.E_tot, w.tile_m)
    expect = g2.gemm2_combine(wl.bf16_bits(x.cpu()), wl.bf16_bits(W2), idx, wt, r["inv_perm"])
    got = np.concatenate([o[:len(G.tokens_of_rank(w.T, w.EP, d))] for d, o in enumerate(outs)])
    assert np.max(np.abs(got - expect)) <= G.tolerance(expect)


def test_argument_validation():
    h = G.handle()
    w = wl.TINY
    idx, _, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    ws, idx_d, S = G.build_routing(w, idx, None)
    hr = torch.empty(B.moe_gemm1_workspace_bytes(ws.shape), dtype=torch.uint8, device="cuda")
    x = torch.empty((w.R, w.I), dtype=torch.bfloat16, device="cuda")
    hd, Wd = hidden.cuda(), W1.cuda()
    with pytest.raises(B.MoeError) as e:
        B.moe_gemm1_act(h, hd, Wd, ws.shape, 96, ws.routing, S, hr, x, ws.status)
    assert e.value.code == B.MOE_ERR_UNSUPPORTED
    with pytest.raises(B.MoeError) as e:
        B.moe_gemm1_act(h, hd, Wd, ws.shape, w.tile_m, ws.routing, S, hr, x.data_ptr() + 2, ws.status)
    assert e.value.code == B.MOE_ERR_ALIGN
    bad = B.make_shape(w.T, w.H, w.I + 8, w.E_tot, w.k_tot, w.TP, w.EP, w.L)
    with pytest.raises(B.MoeError) as e:
        B.moe_gemm1_act(h, hd, Wd, bad, w.tile_m, ws.routing, S, hr, x, ws.status)
    assert e.value.code == B.MOE_ERR_SHAPE


@pytest.mark.parametrize("counts_on_device", [False, True], ids=["host_counts", "device_counts"])
def test_post_router_layer_against_the_oracle_chain(counts_on_device):
    # the three operations of Section II-A in one call, against the oracle's GEMM1 + activation (rounded to
    # bf16 as the stored intermediate is) followed by the oracle's GEMM2 + combine
    h = G.handle()
    w = replace(wl.TINY, name="layer3", T=500, E=10, k=3, n_shared=1, H=256, I=256, TP=2, EP=2, L=2,
                tile_m=128, tile_n=128, routing="zipf", zipf_s=1.0, target_r_expert=2.0)
    idx, wt, _ = wl.make_routing(w)
    hidden, W1 = wl.make_gemm1_data(w)
    _, W2 = wl.make_data(w)
    ws = B.alloc_workspace(G.shape_of(w), w.tile_m, w.tile_n)
    hr = torch.empty(B.moe_gemm1_workspace_bytes(ws.shape), dtype=torch.uint8, device="cuda")
    xr = torch.empty((w.R, w.I), dtype=torch.bfloat16, device="cuda")
    idx_d, wt_d = torch.from_numpy(idx).cuda(), torch.from_numpy(wt).cuda()
    for o in ws.out:
        o.fill_(float("nan"))
    plan = B.moe_post_router_layer(h, hidden.cuda(), W1.cuda(), W2.cuda(), idx_d, wt_d, ws, hr, xr,
                                   counts_on_device=counts_on_device)
    torch.cuda.synchronize()
    assert B.moe_get_status(h, ws.status).code == 0 and plan.comm_ctas >= 1
    r = rr.build_routing(idx, w.E_tot, w.tile_m)
    x_ref = g1.gemm1_act(wl.bf16_bits(hidden), wl.bf16_bits(W1), idx, r["perm"])
    x_bits = wl.bf16_bits(torch.from_numpy(x_ref).bfloat16())
    expect = g2.gemm2_combine(x_bits, wl.bf16_bits(W2), idx, wt, r["inv_perm"])
    outs = [o.float().cpu().numpy() for o in ws.out]
    got = np.concatenate([o[:len(G.tokens_of_rank(w.T, w.EP, d))] for d, o in enumerate(outs)])
    assert not np.isnan(got).any()
    # the intermediate may differ from the oracle's by one bf16 step in a few places: same tolerance form
    assert np.max(np.abs(got - expect)) <= G.tolerance(expect)


def test_random_small_shapes_against_the_oracle():
    # seeded fuzz: ragged token counts, partial k-blocks and n-tiles, every m-tile size, empty experts
    rng = np.random.default_rng(77)
    for case in range(14):
        tile_m = int(rng.choice([64, 128, 256]))
        w = replace(wl.TINY, name=f"g1fuzz{case}", T=int(rng.choice([1, 9, 130, 257, 600])),
                    H=int(rng.choice([64, 80, 144, 256, 528])), I=int(rng.choice([16, 48, 128, 144, 272])),
                    E=int(rng.integers(1, 24)), k=1, n_shared=int(rng.choice([0, 1])), TP=1, EP=1, L=1,
                    tile_m=tile_m, tile_n=256 if tile_m == 256 else 64, routing_seed=300 + case, data_seed=400 + case)
        w = replace(w, k=int(rng.integers(1, min(w.E, 3) + 1)))
        _check(w, counts_on_device=bool(rng.integers(2)))


@pytest.mark.parametrize("tile_m", [64, 128, 256])
@pytest.mark.parametrize("H,I", [(64, 16), (272, 208), (1024, 128)], ids=str)
def test_row_gather_at_the_edges_of_the_m_tiles(tile_m, H, I):
    # experts with 1, 3, 4, 5, 127 ... 257 rows: whole and partial groups of rows, m-tiles whose second half is empty,
    # holds one row, is full; shapes with one k-block, a partial one, and more than the operand ring holds
    counts = [1, 3, 4, 5, 127, 128, 129, 0, 255, 256, 257]
    idx = np.repeat(np.arange(len(counts)), counts).astype(np.int32)
    idx = np.random.default_rng(0).permutation(idx)[:, None].copy()
    w = replace(wl.TINY, name="gather", T=len(idx), E=len(counts), k=1, H=H, I=I, tile_m=tile_m, tile_n=256 if tile_m == 256 else 64,
                TP=1, EP=1, L=1, data_seed=5)
    hidden, W1 = wl.make_gemm1_data(w)
    x, _ = _run(w, idx, hidden, W1, counts_on_device=True)
    r = rr.build_routing(idx, w.E_tot, w.tile_m)
    ref = g1.gemm1_act(wl.bf16_bits(hidden), wl.bf16_bits(W1), idx, r["perm"], rows=np.arange(w.R, dtype=np.int32))
    got = x.float().cpu().numpy()
    assert not np.isnan(got).any()
    assert np.all(np.abs(got - ref) <= _tolerance(ref)), float(np.max(np.abs(got - ref)))


@pytest.mark.parametrize("T,I", [(4, 1408), (4, 1376), (7, 1408), (10, 1408)], ids=str)
def test_tile_widths_of_the_smallest_batches(T, I):
    # up to 8 / 14 / 20 m-tiles: 96-column tiles (the last one whole, then 32 columns wide), 128-column ones in one wave and in two
    w = replace(wl.TINY, name="narrow", T=T, E=40, k=2, H=320, I=I, tile_m=128, tile_n=64, TP=1, EP=1, L=1)
    _check(w, counts_on_device=True)
    _check(replace(w, I=176), counts_on_device=False)      # 64-column tiles


@pytest.mark.parametrize("tile_m,E", [(128, 148), (128, 149), (128, 296), (128, 297), (256, 73), (256, 74), (256, 75), (256, 149)], ids=str)
def test_tiles_dealt_by_whole_waves(tile_m, E):
    # one m-tile per expert, one tile each: a wave of 148 CTAs (74 pairs), one tile more, two waves, one more
    w = replace(wl.TINY, name="waves", T=8 * E, E=E, k=2, H=256, I=128, tile_m=tile_m, tile_n=256, TP=1, EP=1, L=1)
    idx, _, _ = wl.make_routing(w)
    assert rr.build_routing(idx, E, tile_m)["S"] == E
    _check(w, n_rows=200, counts_on_device=True)


@pytest.mark.parametrize("tile_m,tile_n", [(64, 64), (128, 128), (256, 256)], ids=str)
@pytest.mark.parametrize("I", [16, 80, 144], ids=str)     # one group of columns, a tile that ends in its first half, in its second tile
def test_row_counts_around_the_steps_of_the_mma(tile_m, tile_n, I):
    # an m-tile is computed for its rows, rounded up to 16 (a pair: 32, half of them in each CTA)
    counts = [8, 9, 15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 95, 97, 159, 161, 223, 225, 0, 2]
    idx = np.repeat(np.arange(len(counts)), counts).astype(np.int32)
    idx = np.random.default_rng(3).permutation(idx)[:, None].copy()
    w = replace(wl.TINY, name="rowsteps", T=len(idx), E=len(counts), k=1, H=144, I=I, tile_m=tile_m, tile_n=tile_n, TP=1, EP=1, L=1, data_seed=6)
    _check(w, counts_on_device=True)
