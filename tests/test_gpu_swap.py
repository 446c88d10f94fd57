"""Residual swap-in (Section "Multi-Tenant Serving": only the residual moves
host -> device): ordering against applies, stale segments, blob checks."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_close, oracle_tables

pytestmark = pytest.mark.gpu


def _workload(wl):
    T = 48
    u = (wl.uniform(31, 1, T) * 6).astype(np.int32)
    return wl.Workload("swap", 31, [("p", 256, 384)], 2, [16, 16], 8, [2] * 8, dom_ids=u % 2, slot_ids=u)


def _oracle(oracle_mod, w, version_of):
    cents, res = oracle_tables(w, 0, version=version_of)
    return oracle_mod.apply(w.x(0), w.y_in(0), w.dom_ids, w.slot_ids, cents, res)


def test_reload_between_batches_on_side_stream(salt_lib, oracle_mod, wl):
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    w = _workload(wl)
    side = torch.cuda.Stream()
    comp = torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        x = bf16_tensor(w.x(0))
        y1 = bf16_tensor(w.y_in(0))
        y2 = bf16_tensor(w.y_in(0))
        r.build(stream=comp)
        salt.salt_lora_apply(r.ctx, r.seg, 0, x, y1, comp)
        # swap new residuals into slots 1 and 3 while the first apply may still run
        b1 = r.make_blob(1, version=7)
        b3 = r.make_blob(3, version=7)
        salt.salt_residual_load(r.ctx, 1, b1, side)
        salt.salt_residual_load(r.ctx, 3, b3, side)
        with pytest.raises(salt.SaltError) as e:  # the built batch names slots 1 and 3
            salt.salt_lora_apply(r.ctx, r.seg, 0, x, y2, comp)
        assert e.value.name == "SALT_ERR_STALE_SEGMENTS"
        r.build(stream=comp)  # waits for the swaps of the slots it names
        salt.salt_lora_apply(r.ctx, r.seg, 0, x, y2, comp)
        torch.cuda.synchronize()
        assert r.device_error() == 0
        got1, got2 = bf16_bits(y1), bf16_bits(y2)
    assert_close(got1, _oracle(oracle_mod, w, lambda u: 0), "before the swap")
    assert_close(got2, _oracle(oracle_mod, w, lambda u: 7 if u in (1, 3) else 0), "after the swap")


def test_unreferenced_slot_load_keeps_segments_valid(salt_lib, oracle_mod, wl):
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    w = _workload(wl)
    w.slot_ids = np.where(w.slot_ids == 7, 6, w.slot_ids).astype(np.int32)  # slot 7 unused
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        r.build()
        salt.salt_residual_load(r.ctx, 7, r.make_blob(7, version=3), torch.cuda.Stream())
        x = bf16_tensor(w.x(0))
        y = bf16_tensor(w.y_in(0))
        salt.salt_lora_apply(r.ctx, r.seg, 0, x, y)  # no stale error: slot 7 is not named
        torch.cuda.synchronize()
        got = bf16_bits(y)
    assert_close(got, _oracle(oracle_mod, w, lambda u: 0), "unrelated swap")


def test_apply_on_another_stream_waits_for_the_build(salt_lib, oracle_mod, wl):
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    w = _workload(wl)
    s_build, s_apply = torch.cuda.Stream(), torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        x = bf16_tensor(w.x(0))
        y = bf16_tensor(w.y_in(0))
        torch.cuda.synchronize()
        r.build(stream=s_build)
        salt.salt_lora_apply(r.ctx, r.seg, 0, x, y, s_apply)
        torch.cuda.synchronize()
        got = bf16_bits(y)
    assert_close(got, _oracle(oracle_mod, w, lambda u: 0), "cross-stream")


def test_blob_checks(salt_lib, wl):
    from paper_2608_03579_gb300.runner import SaltRunner
    salt = salt_lib
    w = _workload(wl)
    with SaltRunner(w) as r:
        good = r.make_blob(0)
        # pageable host memory is refused
        with pytest.raises(salt.SaltError) as e:
            salt.salt_residual_load(r.ctx, 0, good.numpy().copy(), None)
        assert e.value.name == "SALT_ERR_NOT_PINNED_HOST"
        # wrong magic
        bad = good.clone().pin_memory()
        bad[0] ^= 0xFF
        with pytest.raises(salt.SaltError) as e:
            salt.salt_residual_load(r.ctx, 0, bad, None)
        assert e.value.name == "SALT_ERR_BAD_BLOB"
        # a blob packed for another layer table
        other = torch.empty(salt.salt_residual_blob_bytes([256], [392], 2), dtype=torch.uint8, pin_memory=True)
        salt.salt_residual_blob_pack([256], [392], 2, 1.0, np.zeros(512, np.uint16), np.zeros(784, np.uint16),
                                     other.numpy(), other.numel())
        with pytest.raises(salt.SaltError) as e:
            salt.salt_residual_load(r.ctx, 0, other, None)
        assert e.value.name == "SALT_ERR_BAD_BLOB"
        # rank above the context's r_max (2)
        big = r.make_blob(0, rank=3)
        with pytest.raises(salt.SaltError) as e:
            salt.salt_residual_load(r.ctx, 0, big, None)
        assert e.value.name == "SALT_ERR_RANK"
        with pytest.raises(salt.SaltError) as e:
            salt.salt_residual_load(r.ctx, 8, good, None)
        assert e.value.name == "SALT_ERR_SLOT_RANGE"


def test_huge_page_host_blob_swap(salt_lib, oracle_mod, wl):
    # salt_host_alloc memory is page-locked: a blob packed into it swaps in
    # asynchronously and the apply reads the new residual.
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    w = _workload(wl)
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        nb = r.blob_bytes(2)
        hb = salt.salt_host_alloc(3 * nb + 1000)
        try:
            assert hb.nbytes == 3 * nb + 1000 and int(hb.tensor[:4096].sum()) == 0
            blob = hb.tensor[nb:2 * nb]
            r.make_blob(2, version=5, out=blob)
            side = torch.cuda.Stream()
            salt.salt_residual_load(r.ctx, 2, blob, side)
            r.build()
            x = bf16_tensor(w.x(0))
            y = bf16_tensor(w.y_in(0))
            salt.salt_lora_apply(r.ctx, r.seg, 0, x, y)
            torch.cuda.synchronize()
            got = bf16_bits(y)
        finally:
            hb.close()
    assert_close(got, _oracle(oracle_mod, w, lambda u: 5 if u == 2 else 0), "huge-page host blob")


def test_batch_load_between_batches_on_side_stream(salt_lib, oracle_mod, wl):
    """salt_residual_load_batch: the same ordering as single loads (the swap
    waits for the applies that read the slots, the segments turn stale, a
    rebuild waits for the copies), one call for several slots; a bad blob in
    the batch loads nothing."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    w = _workload(wl)
    side = torch.cuda.Stream()
    comp = torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        x = bf16_tensor(w.x(0))
        y1 = bf16_tensor(w.y_in(0))
        y2 = bf16_tensor(w.y_in(0))
        y3 = bf16_tensor(w.y_in(0))
        r.build(stream=comp)
        salt.salt_lora_apply(r.ctx, r.seg, 0, x, y1, comp)
        # one blob from a huge-page region of the library, two from torch's pinned memory
        nb = r.blob_bytes(2)
        region = salt.salt_host_alloc(nb)
        try:
            b0 = r.make_blob(0, version=5, out=region.tensor[:nb])
            b2 = r.make_blob(2, version=5)
            b5 = r.make_blob(5, version=5)
            # a batch holding one bad blob is refused before anything is enqueued
            bad = r.make_blob(4, version=5).clone().pin_memory()
            bad[0] ^= 0xFF  # magic
            with pytest.raises(salt.SaltError):
                salt.salt_residual_load_batch(r.ctx, [0, 4], [b0, bad], side)
            salt.salt_lora_apply(r.ctx, r.seg, 0, x, y2, comp)  # still valid: nothing was loaded
            salt.salt_residual_load_batch(r.ctx, [0, 2, 5], [b0, b2, b5], side)
            with pytest.raises(salt.SaltError) as e:
                salt.salt_lora_apply(r.ctx, r.seg, 0, x, y3, comp)
            assert e.value.name == "SALT_ERR_STALE_SEGMENTS"
            r.build(stream=comp)
            salt.salt_lora_apply(r.ctx, r.seg, 0, x, y3, comp)
            torch.cuda.synchronize()
            assert r.device_error() == 0
            got1, got2, got3 = bf16_bits(y1), bf16_bits(y2), bf16_bits(y3)
        finally:
            torch.cuda.synchronize()
            salt.salt_host_free(region)
    assert_close(got1, _oracle(oracle_mod, w, lambda u: 0), "before the batch")
    assert_close(got2, _oracle(oracle_mod, w, lambda u: 0), "after the refused batch")
    assert_close(got3, _oracle(oracle_mod, w, lambda u: 5 if u in (0, 2, 5) else 0), "after the batch")


@pytest.mark.parametrize("slots,shift", [
    ([0, 1, 2, 3, 4, 5], 0),   # one launch
    ([6, 1, 3, 0, 5], 0),      # the same, slots in no order
    ([6, 1, 3, 0, 5], 8),      # blobs off the 16-byte boundaries: copies
    ([2, 1, 3, 2, 5], 0),      # a slot named twice: copies, the last one stays
])
def test_batch_load_from_a_host_region(salt_lib, oracle_mod, wl, slots, shift):
    """Batches the swap kernel takes and ones it must not: ranks 1 and 2, blob
    sizes that are no multiple of a CTA's piece, each slot loaded twice."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt = salt_lib
    T = 48
    u = (wl.uniform(31, 1, T) * 8).astype(np.int32) % 8
    w = wl.Workload("swap_region", 31, [("p", 2056, 384), ("q", 4096, 1032)], 2, [16, 16], 8, [1, 2] * 4, dom_ids=u % 2,
                    slot_ids=u)
    side, comp = torch.cuda.Stream(), torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        step = (r.blob_bytes(2) + 255) // 256 * 256
        region = salt.salt_host_alloc(2 * len(slots) * step + 256)
        try:
            y = {}
            for turn in range(2):
                blobs = []
                for i, sl in enumerate(slots):
                    nb, at = r.blob_bytes(w.r_u[sl]), (turn * len(slots) + i) * step + shift
                    blobs.append(r.make_blob(sl, version=10 * turn + i + 1, out=region.tensor[at:at + nb]))
                r.build(stream=comp)
                salt.salt_residual_load_batch(r.ctx, slots, blobs, side)
                r.build(stream=comp)
                xs = bf16_tensor(w.x(1))
                y[turn] = bf16_tensor(w.y_in(1))
                salt.salt_lora_apply(r.ctx, r.seg, 1, xs, y[turn], comp)
            torch.cuda.synchronize()
            assert r.device_error() == 0
            assert salt.salt_guard_check(r.ctx, r.seg) == 0
        finally:
            torch.cuda.synchronize()
            salt.salt_host_free(region)
    for turn in range(2):
        last = {sl: 10 * turn + i + 1 for i, sl in enumerate(slots)}
        cents, res = oracle_tables(w, 1, version=lambda v: last.get(v, 0))
        ref = oracle_mod.apply(w.x(1), w.y_in(1), w.dom_ids, w.slot_ids, cents, res)
        assert_close(bf16_bits(y[turn]), ref, f"swap {turn} of {slots}")


@pytest.mark.parametrize("layers,n_slots,kind", [
    ([("p", 64, 64)], 300, "many"),                  # more blobs than a launch holds: two launches, one event
    ([("p", 256, 264)] * 2, 6, "outside"),           # one blob in other pinned memory: copies
    ([("p", 8192, 8192)] * 48, 4, "large"),          # blobs of 3 MiB and a header: copies
    ([("p", 8192, 8192)] * 47, 4, "below large"),    # the largest of such layers below: one launch
])
def test_batch_load_limits(salt_lib, oracle_mod, wl, layers, n_slots, kind):
    """Batches at the limits of the swap kernel: every slot holds its blob."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt, l = salt_lib, len(layers) - 1
    u = np.arange(2 * n_slots, dtype=np.int32) % n_slots
    w = wl.Workload("swap_limits", 43, layers, 1, [1], n_slots, [2] * n_slots, dom_ids=np.zeros_like(u), slot_ids=u)
    side, comp = torch.cuda.Stream(), torch.cuda.Stream()
    with SaltRunner(w) as r:
        assert (kind == "large") == (r.blob_bytes(2) > 3 << 20)
        r.pin_centroids()
        step = (r.blob_bytes(2) + 255) // 256 * 256
        region = salt.salt_host_alloc(n_slots * step)
        try:
            blobs = [r.make_blob(v, out=None if kind == "outside" and v == 3 else
                                 region.tensor[v * step:v * step + r.blob_bytes(2)]) for v in range(n_slots)]
            salt.salt_residual_load_batch(r.ctx, list(range(n_slots)), blobs, side)
            r.build(stream=comp)
            x, y = bf16_tensor(w.x(l)), bf16_tensor(w.y_in(l))
            salt.salt_lora_apply(r.ctx, r.seg, l, x, y, comp)
            torch.cuda.synchronize()
            assert r.device_error() == 0
            assert salt.salt_guard_check(r.ctx, r.seg) == 0
        finally:
            torch.cuda.synchronize()
            salt.salt_host_free(region)
    cents, res = oracle_tables(w, l)
    ref = oracle_mod.apply(w.x(l), w.y_in(l), w.dom_ids, w.slot_ids, cents, res)
    assert_close(bf16_bits(y), ref, f"batch load, {kind}")


def test_batch_events_are_used_again(salt_lib, oracle_mod, wl):
    """Batches of which single loads and smaller batches replace a part: a
    batch's event may be recorded again only once no slot's last load is that
    batch.  Every batch is followed at once by a build and an apply that read
    every slot; blobs large enough that a missed wait reads an old one."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt, n = salt_lib, 10
    u = np.arange(40, dtype=np.int32) % n
    w = wl.Workload("swap_events", 44, [("p", 256, 264)] + [("q", 8192, 8192)] * 12 + [("o", 264, 256)], 1, [1], n, [2] * n,
                    dom_ids=np.zeros_like(u), slot_ids=u)
    l = len(w.layers) - 1
    # the event each is recorded in, and which others still hold a slot (event 0: the set-up's load of all ten)
    turns = [[0, 1, 2, 3, 4, 5],   # 1; 0 keeps 6-9
             [2],                  # the slot's own; 1 keeps 0 1 3 4 5
             [6, 7, 8, 9],         # 2; then 0 is free
             [0, 1, 3, 4],         # 0 again; 1 keeps 5
             [5, 6, 7, 8, 9],      # 3; then 1 and 2 are free
             [0, 1, 2, 3],         # 1 again; 0 keeps 4
             [4, 5, 6, 7],         # 2 again; then 0 is free, 3 keeps 8 9
             [8, 9, 0, 4],         # 0 again; then 3 is free
             [1, 2, 3, 5, 6, 7]]   # 3 again
    side, comp = torch.cuda.Stream(), torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        step = (r.blob_bytes(2) + 255) // 256 * 256
        region = salt.salt_host_alloc((n + sum(map(len, turns))) * step)
        at = iter(range(0, region.nbytes, step))

        def blob(slot, version):
            a = next(at)
            return r.make_blob(slot, version, out=region.tensor[a:a + r.blob_bytes(2)])

        try:
            salt.salt_residual_load_batch(r.ctx, list(range(n)), [blob(v, 0) for v in range(n)], side)
            side.synchronize()
            blobs = [[blob(v, t + 1) for v in slots] for t, slots in enumerate(turns)]
            x = bf16_tensor(w.x(l))
            ys = [bf16_tensor(w.y_in(l)) for _ in turns]
            torch.cuda.synchronize()
            for slots, bl, y in zip(turns, blobs, ys):
                salt.salt_residual_load_batch(r.ctx, slots, bl, side)
                r.build(stream=comp)
                salt.salt_lora_apply(r.ctx, r.seg, l, x, y, comp)
            torch.cuda.synchronize()
            assert r.device_error() == 0
            assert salt.salt_guard_check(r.ctx, r.seg) == 0
        finally:
            torch.cuda.synchronize()
            salt.salt_host_free(region)
    last = {v: 0 for v in range(n)}
    for t, (slots, y) in enumerate(zip(turns, ys)):
        last.update({v: t + 1 for v in slots})
        cents, res = oracle_tables(w, l, version=lambda v: last[v])
        ref = oracle_mod.apply(w.x(l), w.y_in(l), w.dom_ids, w.slot_ids, cents, res)
        assert_close(bf16_bits(y), ref, f"after batch {t}")


def test_batch_load_beside_base_calls(salt_lib, oracle_mod, wl):
    """The swap kernel on a side stream while the base kernel runs (both fit an
    SM): base results are those without it, and the slots hold their blobs."""
    from paper_2608_03579_gb300.runner import SaltRunner, bf16_bits, bf16_tensor
    salt, T, n = salt_lib, 256, 8
    u = (wl.uniform(45, 1, T) * n).astype(np.int32) % n
    w = wl.Workload("swap_base", 45, [("p", 1032, 2048)] + [("q", 8192, 8192)] * 20, 2, [16, 16], 2 * n, [2] * (2 * n),
                    dom_ids=u % 2, slot_ids=u)
    side, comp = torch.cuda.Stream(), torch.cuda.Stream()
    with SaltRunner(w) as r:
        r.pin_centroids()
        r.load_slots()
        step = (r.blob_bytes(2) + 255) // 256 * 256
        region = salt.salt_host_alloc(n * step)
        try:
            blobs = [r.make_blob(n + i, 5, out=region.tensor[i * step:i * step + r.blob_bytes(2)]) for i in range(n)]
            W = bf16_tensor(wl.normal_bf16(45, wl.stream_id(wl.K_AUX, 41), 1032 * 2048, 1032 ** -0.5).reshape(2048, 1032))
            x, y0 = bf16_tensor(w.x(0)), bf16_tensor(w.y_in(0))
            ys = [torch.empty(T, 2048, dtype=torch.bfloat16, device="cuda") for _ in range(24)]
            r.build(stream=comp)
            torch.cuda.synchronize()
            for i, y in enumerate(ys):
                if i == 2:
                    salt.salt_residual_load_batch(r.ctx, list(range(n, 2 * n)), blobs, side)
                salt.salt_lora_apply_with_base(r.ctx, r.seg, 0, x, W, 1, y, comp)
            r.build(slot=w.slot_ids + n, stream=comp)
            salt.salt_lora_apply(r.ctx, r.seg, 0, x, y0, comp)
            torch.cuda.synchronize()
            assert r.device_error() == 0
            assert salt.salt_guard_check(r.ctx, r.seg) == 0
        finally:
            torch.cuda.synchronize()
            salt.salt_host_free(region)
    first = bf16_bits(ys[0])
    assert all(np.array_equal(first, bf16_bits(y)) for y in ys[1:])
    cents, res = oracle_tables(w, 0, version=lambda v: 5 if v >= n else 0)
    ref = oracle_mod.apply(w.x(0), w.y_in(0), w.dom_ids, w.slot_ids + n, cents, res)
    assert_close(bf16_bits(y0), ref, "slots loaded beside base calls")
