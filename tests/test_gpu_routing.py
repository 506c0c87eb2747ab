"""GPU routing builder against the routing reference: every array bit-exact."""

import numpy as np
import pytest
import torch

from oracle import routing_ref as rr
from paper_2609_07536_b200 import binding as B
from paper_2609_07536_b200 import workloads as wl
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

KEYS = ["counts", "offsets", "tiles", "tile_offsets", "perm", "inv_perm", "pad_row",
        "mtile_expert", "mtile_first_row", "mtile_valid"]


def _compare(w, idx):
    ws, _, S = G.build_routing(w, idx)
    st = B.moe_get_status(G.handle(), ws.status)
    assert st.code == 0
    ref = rr.build_routing(idx, w.E_tot, w.tile_m)
    assert S == ref["S"]
    got = G.routing_to_numpy(ws, S)
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k
    assert ws.tile_counts[:w.E_tot].tolist() == ref["tiles"].tolist()


@pytest.mark.parametrize("w", [wl.TINY, wl.GRANITE, wl.QWEN, wl.DSV2L], ids=lambda w: w.name)
def test_configs(w):
    idx, _, _ = wl.make_routing(w)
    _compare(w, idx)


def test_adversarial():
    from dataclasses import replace
    base = replace(wl.TINY, T=300, E=9, k=1, tile_m=64)
    # one hot expert, others empty
    _compare(base, np.full((300, 1), 4, dtype=np.int32))
    # E = 1
    _compare(replace(base, E=1), np.zeros((300, 1), dtype=np.int32))
    # T not a tile multiple, k = 3, tile 128, many empty experts
    rng = np.random.default_rng(0)
    w = replace(wl.TINY, T=1001, E=70, k=3, tile_m=128)
    idx = np.stack([rng.choice(13, 3, replace=False) * 5 for _ in range(1001)]).astype(np.int32)
    _compare(w, idx)
    # a single token
    _compare(replace(base, T=1, E=4, k=2), np.array([[3, 0]], dtype=np.int32))
    # the sweep's largest size
    big = wl.sweep_workloads(T_list=(32768,), s_list=(1.2,), EP_list=(4,), tiles=((128, 256),))[0]
    idx, _, _ = wl.make_routing(big)
    _compare(big, idx)


def test_batches_of_the_cluster_launch():
    """33 to 128 chunks of 256 assignments go through one cluster of 8 CTAs: uneven chunk runs (a CTA with
    fewer chunks, a CTA with none), a ragged last chunk, one hot expert, bad ids reported."""
    from dataclasses import replace
    rng = np.random.default_rng(3)
    for T, E, k, tm in ((2817, 40, 3, 128),      # 8451 assignments: 34 chunks, CTA 7 of 8 gets none
                        (9003, 66, 1, 64),       # 36 chunks, the last one ragged
                        (4099, 256, 8, 256),     # 129 chunks: the first size of the four-launch path
                        (4000, 200, 8, 128)):    # 125 chunks, many experts
        w = replace(wl.TINY, T=T, E=E, k=k, tile_m=tm, tile_n=256 if tm == 256 else 64)
        idx = np.stack([rng.choice(E, k, replace=False) for _ in range(T)]).astype(np.int32)
        _compare(w, idx)
    w = replace(wl.TINY, T=10000, E=9, k=1, tile_m=64)
    _compare(w, np.full((10000, 1), 4, dtype=np.int32))
    idx = rng.integers(0, 9, size=(10000, 1)).astype(np.int32)
    bad = idx.copy()
    bad[9000, 0] = -3
    ws, _, S = G.build_routing(w, bad)
    st = B.moe_get_status(G.handle(), ws.status, check=False)
    assert st.code == B.MOE_DEV_OOB and st.detail == 9000
    _compare(w, idx)


def test_bad_ids_are_reported_not_fatal():
    from dataclasses import replace
    w = replace(wl.TINY, T=64, E=8, k=2)
    idx, _, _ = wl.make_routing(w)
    bad = idx.copy()
    bad[5, 1] = 99
    ws, _, S = G.build_routing(w, bad)
    st = B.moe_get_status(G.handle(), ws.status, check=False)
    assert st.code == B.MOE_DEV_OOB and st.detail == 5 * 2 + 1
    dup = idx.copy()
    dup[7, 1] = dup[7, 0]
    ws, _, S = G.build_routing(w, dup)
    st = B.moe_get_status(G.handle(), ws.status, check=False)
    assert st.code == B.MOE_DEV_DUP_EXPERT and st.detail == 7
    # the context is still usable
    _compare(w, idx)


@pytest.mark.parametrize("T,E,k", [
    (128, 66, 8), (1025, 9, 1),          # 1024 and 1025 assignments: one CTA, the first cluster of two
    (683, 33, 3), (1366, 65, 3),         # 2049 and 4098: clusters of four and eight, tokens straddle the rows of 32
    (8193, 1, 1), (2341, 1000, 7),       # 8193 and 16387: sixteen CTAs, one row and two rows per warp
    (16384, 66, 8), (18725, 40, 7),      # 131072, and 131075: the first size of the four launches
], ids=lambda v: str(v))
def test_edges_of_the_one_launch_build(T, E, k):
    from dataclasses import replace
    rng = np.random.default_rng(T)
    idx = np.argsort(rng.random((T, E), dtype=np.float32), axis=1)[:, :k].astype(np.int32)
    _compare(replace(wl.TINY, T=T, E=E, k=k, tile_m=64), idx)


@pytest.mark.parametrize("t,slots", [(3, (0, 2)), (10, (0, 2)), (10, (1, 2)), (341, (0, 1)), (682, (0, 2))])
def test_repeated_experts_are_found_across_the_rows_of_a_warp(t, slots):
    # k = 3: token 10 holds assignments 30, 31 | 32, token 341 1023 | 1024 (the next CTA's first row)
    from dataclasses import replace
    w = replace(wl.TINY, T=700, E=8, k=3)
    idx = np.tile(np.array([[1, 5, 7]], dtype=np.int32), (700, 1))
    idx[t, slots[1]] = idx[t, slots[0]]
    ws, _, _ = G.build_routing(w, idx)
    st = B.moe_get_status(G.handle(), ws.status, check=False)
    assert (st.code, st.detail, st.count) == (B.MOE_DEV_DUP_EXPERT, t, 1)


@pytest.mark.parametrize("T,E,k", [
    (1, 1, 1), (11, 3, 3),                  # less than one row of 32, a row and a bit
    (682, 33, 3), (683, 33, 3),             # 2046 assignments, and 2049: built by a launch of its own
    (256, 512, 8), (256, 513, 8),           # 2048, at and above the expert limit of GEMM1
    (200, 640, 7), (200, 641, 7),           # at and above that of the fused kernel
], ids=lambda v: str(v))
@pytest.mark.parametrize("entry", ["layer", "post_router"])
def test_routing_built_by_the_kernel_that_uses_it(entry, T, E, k):
    from dataclasses import replace
    h = G.handle()
    w = replace(wl.TINY, T=T, E=E, k=k, H=128, I=64, tile_m=64, tile_n=128, TP=1, EP=1, L=1)
    rng = np.random.default_rng(T + E)
    idx = np.argsort(rng.random((T, E), dtype=np.float32), axis=1)[:, :k].astype(np.int32)
    x = torch.zeros(T * k, 64, dtype=torch.bfloat16, device="cuda")
    hidden = torch.ones(T, 128, dtype=torch.bfloat16, device="cuda")
    W1, W2 = (torch.zeros(E, *s, dtype=torch.bfloat16, device="cuda") for s in ((2, 64, 128), (128, 64)))
    wt = torch.ones(T, k, device="cuda")
    ws = B.alloc_workspace(G.shape_of(w), w.tile_m, w.tile_n)
    hr = torch.empty(B.moe_gemm1_workspace_bytes(ws.shape), dtype=torch.uint8, device="cuda")

    def run(ids, on_device):
        ws.routing_ws.fill_(0x77)
        ws.tile_counts.fill_(-7)
        B.moe_clear_status(h, ws.status)
        d = torch.from_numpy(np.ascontiguousarray(ids)).cuda()
        if entry == "layer":
            B.moe_layer(h, x, W2, d, wt, ws, counts_on_device=on_device)
        else:
            B.moe_post_router_layer(h, hidden, W1, W2, d, wt, ws, hr, x, counts_on_device=on_device)
        torch.cuda.synchronize()
        return B.moe_get_status(h, ws.status, check=False)

    ref = rr.build_routing(idx, E, w.tile_m)
    for on_device in (False, True):
        assert run(idx, on_device).code == 0
        got = G.routing_to_numpy(ws, ref["S"])
        for key in KEYS:
            assert np.array_equal(got[key], ref[key]), (key, on_device)
        assert on_device or ws.tile_counts.tolist() == ref["tiles"].tolist() + [ref["S"]]
    bad = idx.copy()
    bad[T // 2, k - 1] = E
    st = run(bad, False)                    # reported once, whatever the number of CTAs
    assert (st.code, st.detail, st.count) == (B.MOE_DEV_OOB, T // 2 * k + k - 1, 1)
    if k > 1:
        dup = idx.copy()
        dup[T // 2, k - 1] = dup[T // 2, 0]
        st = run(dup, False)
        assert (st.code, st.detail, st.count) == (B.MOE_DEV_DUP_EXPERT, T // 2, 1)


@pytest.mark.parametrize("T,E,k", [(5, 33, 2), (40000, 40, 4)], ids=["one_launch", "four_launches"])
@pytest.mark.parametrize("pinned", [True, False], ids=["pinned", "pageable"])
def test_counts_reach_any_host_memory(T, E, k, pinned):
    from dataclasses import replace
    w = replace(wl.TINY, T=T, E=E, k=k, tile_m=128)
    idx = np.argsort(np.random.default_rng(5).random((T, E), dtype=np.float32), axis=1)[:, :k].astype(np.int32)
    ref = rr.build_routing(idx, E, w.tile_m)
    ws = B.alloc_workspace(G.shape_of(w), w.tile_m, w.tile_n)
    host = torch.full((E + 3,), -7, dtype=torch.int32)
    host = host.pin_memory() if pinned else host
    ws.tile_counts = host[1:E + 2]
    G.build_routing(w, idx, ws)
    assert host.tolist() == [-7] + ref["tiles"].tolist() + [ref["S"], -7]
