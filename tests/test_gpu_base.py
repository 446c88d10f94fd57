"""salt_lora_apply_with_base: the base-weight GEMM fused with the SALT delta
(y = x W_base + s_c (x A_c) B_c + s_u (x a_u) b_u, y written), against the
fp64 oracle's W_final evaluation, for both weight layouts."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_close, guarded_like, guards_intact, oracle_tables

pytestmark = pytest.mark.gpu


def _weight(wl, seed, d_in, d_out, layout):
    W = wl.normal_bf16(seed, wl.stream_id(wl.K_AUX, 40, d_in, d_out), d_in * d_out, 1.0 / np.sqrt(d_in))
    W = W.reshape(d_in, d_out)
    return W if layout == 0 else np.ascontiguousarray(W.T)


def _run(salt, r, w, l, W, layout):
    from paper_2608_03579_gb300.runner import bf16_bits, bf16_tensor
    x = bf16_tensor(w.x(l))
    Wd = bf16_tensor(W)
    y0 = torch.full((w.T, int(w.d_out[l])), float("nan"), dtype=torch.bfloat16, device="cuda")  # never read
    y, buf = guarded_like(y0)
    salt.salt_lora_apply_with_base(r.ctx, r.seg, l, x, Wd, layout, y)
    torch.cuda.synchronize()
    assert guards_intact(buf), "a store ran past y"
    return bf16_bits(y)


def _ref(oracle_mod, w, l, W, layout, rows=None):
    cents, res = oracle_tables(w, l)
    dom = w.dom_ids if rows is None else w.dom_ids[rows]
    slot = w.slot_ids if rows is None else w.slot_ids[rows]
    return oracle_mod.apply(w.x(l), None, w.dom_ids, w.slot_ids, cents, res, rows=rows, w_base=W, w_layout=layout)


@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_config0(salt_lib, oracle_mod, wl, layout):
    from paper_2608_03579_gb300.runner import SaltRunner
    w = wl.config0()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        W = _weight(wl, 0, 512, 512, layout)
        got = _run(salt_lib, r, w, 0, W, layout)
        assert r.device_error() == 0
        assert salt_lib.salt_guard_check(r.ctx, r.seg) == 0
    assert_close(got, _ref(oracle_mod, w, 0, W, layout), f"with base, config 0, layout {layout}")


@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_ragged_and_absent_ids(salt_lib, oracle_mod, wl, layout):
    """d_in, d_out not multiples of the tiles, tokens with no term (x W_base
    alone), a batch that is not a multiple of 128 tokens."""
    from paper_2608_03579_gb300.runner import SaltRunner
    T, n_users = 200, 12
    u = (wl.uniform(21, 1, T) * n_users).astype(np.int32) % n_users
    dom = (u % 3).astype(np.int32)
    slot = u.copy()
    none = wl.uniform(21, 2, T) < 0.2
    dom[none], slot[none] = -1, -1
    dom[wl.uniform(21, 3, T) < 0.1] = -1
    w = wl.Workload("ragged_base", 21, [("p", 72, 520)], 3, [8, 16, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=dom, slot_ids=slot)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        W = _weight(wl, 21, 72, 520, layout)
        got = _run(salt_lib, r, w, 0, W, layout)
        assert r.device_error() == 0
    assert_close(got, _ref(oracle_mod, w, 0, W, layout), f"with base, ragged, layout {layout}")


@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_config3(salt_lib, oracle_mod, wl, layout):
    """One Llama-3.1-8B layer's q (4096 -> 4096) and down (14336 -> 4096) at
    256 decode tokens; rows at every 128-token tile edge, every row block's
    first and last token and a spread sample."""
    from paper_2608_03579_gb300.runner import SaltRunner
    w = wl.config3()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        exp = r.export()
        starts = exp["blocks"][:, 0]
        ends = starts + exp["blocks"][:, 1]
        pos = np.unique(np.concatenate([starts, ends - 1, [0, 127, 128, w.T - 1]]))
        rows = np.unique(np.concatenate([exp["perm"][pos[(pos >= 0) & (pos < w.T)]],
                                         (wl.uniform(3, 77, 24) * w.T).astype(int)]))
        for l in (0, 6):
            W = _weight(wl, 3, int(w.d_in[l]), int(w.d_out[l]), layout)
            got = _run(salt_lib, r, w, l, W, layout)
            assert r.device_error() == 0
            assert_close(got[rows], _ref(oracle_mod, w, l, W, layout, rows=rows),
                         f"with base, config 3 {w.layers[l][0]}, layout {layout}")


ONE, SEVERAL = "one unit a cluster", "several units a cluster"


@pytest.mark.parametrize("T,d_in,d_out,cg,splits,units", [
    (1, 64, 64, 1, False, ONE),           # one token, one K chunk, half a tile of columns
    (24, 4096, 256, 1, True, ONE),        # few tiles: K splits that wait for each other
    (24, 6144, 9728, 1, True, SEVERAL),   # K splits that leave their sums to the last
    (100, 72, 20488, 1, False, SEVERAL),  # one CTA a tile, both accumulators, ring positions across units
    (127, 136, 136, 1, False, ONE), (128, 1032, 392, 1, False, ONE),  # the last batches of one CTA a tile; remainders
    (129, 1032, 392, 2, False, ONE),      # the first batch of CTA pairs: one token in the second half
    (257, 72, 264, 2, False, ONE),        # a second M tile of one token
    (300, 14336, 128, 2, True, ONE),      # K splits of pairs; a second M tile with an empty second half
    (700, 520, 1288, 2, False, ONE),      # more stages than the ring
    (2300, 136, 2056, 2, False, SEVERAL), # several units a pair, a last column tile of 8
])
@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_tile_edges(salt_lib, oracle_mod, wl, layout, T, d_in, d_out, cg, splits, units):
    """Every tile and split shape of the base kernel at its edges (the launch
    shape is checked, so a change of the plan cannot drop one); users in
    random order, stacks of one and of two 64-row chunks, tokens without a
    term; run twice (the split counters must be left at zero)."""
    from paper_2608_03579_gb300.runner import SaltRunner
    n_users = 40
    u = (wl.uniform(31, 1, T) * n_users).astype(np.int32) % n_users
    dom, slot = (u % 2).astype(np.int32), u.copy()
    none = wl.uniform(31, 2, T) < 0.1
    dom[none], slot[none] = -1, -1
    w = wl.Workload("base_edges", 31, [("p", d_in, d_out)], 2, [64, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=dom, slot_ids=slot)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        sh = salt_lib.salt_base_get_shape(r.ctx, r.seg, 0)
        assert (sh["cta_group"], sh["k_splits"] > 1, sh["units"] > sh["clusters"]) == (cg, splits, units == SEVERAL), sh
        W = _weight(wl, 31, d_in, d_out, layout)
        got = _run(salt_lib, r, w, 0, W, layout)
        again = _run(salt_lib, r, w, 0, W, layout)
        assert r.device_error() == 0
        assert salt_lib.salt_guard_check(r.ctx, r.seg) == 0
    assert np.array_equal(got, again)
    rows = np.arange(T) if T < 2000 else np.unique(np.concatenate([np.arange(0, T, 7), [T - 1]]))
    assert_close(got[rows], _ref(oracle_mod, w, 0, W, layout, rows=rows),
                 f"with base, {T} x {d_in} x {d_out}, layout {layout}")


@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_consecutive_and_scattered_tiles(salt_lib, oracle_mod, wl, layout):
    """Long user runs beside users in random order: pairs whose halves are both
    consecutive tokens (x by tile loads), both gathered, and one of each."""
    from paper_2608_03579_gb300.runner import SaltRunner
    u = 2 + (wl.uniform(39, 1, 2240) * 28).astype(np.int32) % 28
    for user, first, n in ((0, 0, 640), (1, 640, 70), (30, 1310, 500), (31, 1810, 128)):
        u[first:first + n] = user
    T, n_users, d_in, d_out = len(u), 32, 520, 776
    w = wl.Workload("base_runs", 39, [("p", d_in, d_out)], 2, [64, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=(u >= 16).astype(np.int32), slot_ids=u)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        perm = r.export()["perm"]
        half = [bool((np.diff(perm[m:m + 128]) == 1).all()) for m in range(0, T - T % 256, 128)]
        kinds = set(zip(half[::2], half[1::2]))
        assert {(True, True), (False, False)} <= kinds and kinds & {(True, False), (False, True)}, kinds
        assert salt_lib.salt_base_get_shape(r.ctx, r.seg, 0)["cta_group"] == 2
        W = _weight(wl, 39, d_in, d_out, layout)
        got = _run(salt_lib, r, w, 0, W, layout)
        assert r.device_error() == 0
        assert salt_lib.salt_guard_check(r.ctx, r.seg) == 0
    assert_close(got, _ref(oracle_mod, w, 0, W, layout), f"with base, consecutive and scattered tiles, layout {layout}")


@pytest.mark.parametrize("layout", [0, 1])
def test_with_base_pairs_repeat(salt_lib, oracle_mod, wl, layout):
    """CTA pairs whose second CTA gathers its rows (users in random order), a
    K loop of several rounds of the ring and delta chunks: every run gives
    the same bits, so no stage is read before the other CTA's copies landed."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    T, n_users, d_in, d_out = 512, 64, 2048, 512
    u = (wl.uniform(33, 1, T) * n_users).astype(np.int32) % n_users
    w = wl.Workload("base_repeat", 33, [("p", d_in, d_out)], 2, [64, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=(u % 2).astype(np.int32), slot_ids=u)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        W = _weight(wl, 33, d_in, d_out, layout)
        x, Wd = bf16_tensor(w.x(0)), bf16_tensor(W)
        ys = [torch.full((T, d_out), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(20)]
        for y in ys:
            salt_lib.salt_lora_apply_with_base(r.ctx, r.seg, 0, x, Wd, layout, y)
        torch.cuda.synchronize()
        assert r.device_error() == 0
    first = bf16_bits(ys[0])
    assert all(np.array_equal(first, bf16_bits(y)) for y in ys[1:])
    assert_close(first, _ref(oracle_mod, w, 0, W, layout), f"with base, repeated, layout {layout}")


@pytest.mark.parametrize("T,d_in,d_out", [(24, 4096, 4096), (24, 8192, 1032), (200, 14336, 2048)])
def test_with_base_splits_on_two_streams(salt_lib, oracle_mod, wl, T, d_in, d_out):
    """K-split launches of two segments objects on two streams: the CTAs of a
    tile need not run together, so every result is the same bits as alone."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt, n_users = salt_lib, 16
    u = (wl.uniform(35, 1, T) * n_users).astype(np.int32) % n_users
    w = wl.Workload("base_streams", 35, [("p", d_in, d_out)], 2, [64, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=(u % 2).astype(np.int32), slot_ids=u)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        segs = [r.seg, salt.salt_segments_create(r.ctx)]
        try:
            for seg in segs:
                salt.salt_build_segments(r.ctx, seg, w.dom_ids, w.slot_ids)
                assert salt.salt_base_get_shape(r.ctx, seg, 0)["k_splits"] > 1
            x, Wd = bf16_tensor(w.x(0)), bf16_tensor(_weight(wl, 35, d_in, d_out, 1))
            ys = [torch.full((T, d_out), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(41)]
            salt.salt_lora_apply_with_base(r.ctx, r.seg, 0, x, Wd, 1, ys[0])
            streams = [torch.cuda.Stream(), torch.cuda.Stream()]
            torch.cuda.synchronize()
            for i, y in enumerate(ys[1:]):
                salt.salt_lora_apply_with_base(r.ctx, segs[i & 1], 0, x, Wd, 1, y, streams[i & 1])
            torch.cuda.synchronize()
            assert r.device_error() == 0
            for seg in segs:
                assert salt.salt_guard_check(r.ctx, seg) == 0
        finally:
            salt.salt_segments_destroy(segs[1])
    first = bf16_bits(ys[0])
    assert all(np.array_equal(first, bf16_bits(y)) for y in ys[1:])
    assert_close(first, _ref(oracle_mod, w, 0, _weight(wl, 35, d_in, d_out, 1), 1), f"two streams, {T} x {d_in} x {d_out}")


@pytest.mark.parametrize("T,later", [
    (40, (17, 1, 0, 40, 41, 500, 11000, 33)),       # one CTA a tile; replayed on up to 86 tiles' worth of tokens
    (300, (130, 257, 20, 300, 301, 8200, 16384, 299)),  # pairs
])
def test_with_base_replayed_after_rebuilds(salt_lib, oracle_mod, wl, T, later):
    """A captured call replayed after rebuilds: batches up to the capture's
    are computed whole, other rows of y stay; a larger one raises a flag and
    leaves y alone, and the next replay is right again."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    n_users, d_in, d_out, T_max = 24, 1032, 392, 16384
    u = (wl.uniform(37, 1, T_max) * n_users).astype(np.int32) % n_users
    w = wl.Workload("base_replay", 37, [("p", d_in, d_out)], 2, [64, 5], n_users, [1, 2] * (n_users // 2),
                    dom_ids=(u % 2).astype(np.int32), slot_ids=u)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        W = _weight(wl, 37, d_in, d_out, 1)
        x, Wd = bf16_tensor(w.x(0)), bf16_tensor(W)
        y = torch.empty(T_max, d_out, dtype=torch.bfloat16, device="cuda")
        s = torch.cuda.Stream()
        r.build(w.dom_ids[:T], w.slot_ids[:T], stream=s)
        salt_lib.salt_lora_apply_with_base(r.ctx, r.seg, 0, x, Wd, 1, y, s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            salt_lib.salt_lora_apply_with_base(r.ctx, r.seg, 0, x, Wd, 1, y, s)
        cents, res = oracle_tables(w, 0)
        for n in later:
            # the last n tokens' ids for the first n tokens: another grouping than at the capture
            dom, slot = w.dom_ids[T_max - n:], w.slot_ids[T_max - n:]
            r.build(dom, slot, stream=s)
            y.fill_(7.0)
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                g.replay()
            torch.cuda.synchronize()
            got = bf16_bits(y)
            assert salt_lib.salt_guard_check(r.ctx, r.seg) == 0
            assert r.device_error() == (0x80 if n > T else 0), n
            done = n if n <= T else 0
            assert (got[done:] == 0x40E0).all(), f"{n} tokens: rows past the batch were written"
            if done:
                ref = oracle_mod.apply(w.x(0)[:n], None, dom, slot, cents, res, w_base=W, w_layout=1)
                assert_close(got[:n], ref, f"captured on {T} tokens, replayed on {n}")


@pytest.mark.parametrize("T,d_out", [(100, 264), (128, 2048), (400, 264), (512, 1032)])
def test_with_base_infinity_stays_in_its_block(salt_lib, oracle_mod, wl, T, d_out):
    """A user whose residual holds infinities: tokens outside the row blocks
    that the user's tokens are in get the values they would without that user."""
    from paper_2608_03579_gb300.runner import SaltRunner
    n_users, d_in, bad = 40, 264, 21
    u = (wl.uniform(47, 1, T) * n_users).astype(np.int32) % n_users
    w = wl.Workload("base_inf", 47, [("p", d_in, d_out)], 4, [64, 5, 16, 64], n_users, [2] * n_users,
                    dom_ids=(u % 4).astype(np.int32), slot_ids=u)
    w.y_mode = "zeros"
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        blob = r.make_blob(bad)
        blob[256 + 2 * 2 * d_in:].view(torch.int16).fill_(0x7F80)  # both rows of B
        salt_lib.salt_residual_load(r.ctx, bad, blob)
        r.build()
        exp = r.export()
        beside = np.zeros(T, bool)
        for start, n, _ in exp["blocks"]:
            tokens = exp["perm"][start:start + n]
            beside[tokens] |= (u[tokens] == bad).any()
        W = _weight(wl, 47, d_in, d_out, 1)
        got = _run(salt_lib, r, w, 0, W, 1)
        assert r.device_error() == 0
    rows = np.flatnonzero(~beside)
    assert 0 < len(rows) < T
    assert_close(got[rows], _ref(oracle_mod, w, 0, W, 1, rows=rows), f"beside an infinity, {T} tokens")
