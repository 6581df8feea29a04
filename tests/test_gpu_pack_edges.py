"""Packing and pruning where their kernels change shape: block widths that are not whole octets beside the operand image,
filter groups narrower than a warp, more taps than a word, more groups than a cluster's shared memory holds, and device
masks that change while a layer is being packed."""
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w_in", ["f32", "bf16"])
@pytest.mark.parametrize("K,C,R,Mb,Nb", [(48, 48, 3, 16, 12), (40, 32, 3, 8, 4), (24, 16, 3, 3, 1), (16, 16, 3, 16, 16), (48, 32, 3, 48, 16),
                                         (272, 64, 3, 16, 32), (32, 32, 6, 16, 16), (64, 16, 7, 4, 2), (160, 96, 1, 32, 48)])
def test_pack_bp_sections_at_the_edges(K, C, R, Mb, Nb, w_in):
    c = inputs.conv_case(N=1, H=8, W=8, C=C, K=K, R=R, S=R, Mb=Mb, Nb=Nb, keep=lambda fb, cb: (3 * fb + 2 * cb) % (R * R + 1), dtype=w_in,
                         act="normal", w_sigma=1.0, seed=1001)
    ref = oracle.pack_bp(c.w, c.tap_mask, Mb, Nb, "bf16")
    w = dev(c.w, w_in)
    assert np.array_equal(npas.pack_bp(w, c.tap_mask, Mb, Nb, torch.bfloat16).data.cpu().numpy(), ref)
    on_gpu = torch.from_numpy(c.tap_mask.view(np.int64)).cuda()
    blob = npas.pack_bp(w, on_gpu, Mb, Nb, torch.bfloat16)
    assert np.array_equal(blob.data.cpu().numpy(), ref)
    assert blob.desc.max_taps == max(1, max(bin(int(v)).count("1") for v in c.tap_mask.ravel()))


@pytest.mark.parametrize("K,C,R,Mb,Nb,w_in", [(3072, 3072, 1, 16, 16, "bf16"), (512, 512, 1, 1, 1, "f32"), (65536, 16, 1, 1, 16, "bf16")])
def test_masks_on_the_device_and_on_the_host_give_the_same_blob(K, C, R, Mb, Nb, w_in):
    """More blocks than the scan keeps counts of; the two ways to pack share no prefix sums."""
    rng = inputs.rng_for(1005)
    w = dev(rng.standard_normal((K, R, R, C), dtype=np.float32), w_in)
    tm = rng.integers(0, 2, (K // Mb, C // Nb)).astype(np.int64)
    on_gpu = npas.pack_bp(w, torch.from_numpy(tm).cuda(), Mb, Nb, torch.bfloat16)
    assert torch.equal(on_gpu.data, npas.pack_bp(w, tm.view(np.uint64), Mb, Nb, torch.bfloat16).data)
    wd, back = npas.unpack_bp(on_gpu)
    assert torch.equal(back.cpu(), torch.from_numpy(tm))


@pytest.mark.parametrize("rate", [1.5, 10.0])
def test_global_pruning_of_more_groups_than_shared_memory_holds(rate):
    """204800 groups over eight CTAs; the scores of one filter block repeat in another, so equal keys meet the budget."""
    rng = inputs.rng_for(1002)
    w = rng.standard_normal((512, 5, 5, 512), dtype=np.float32)
    w[8:16] = w[:8]
    G = (512 // 8) * (512 // 4) * 25
    tm = npas.prune_bp_magnitude_global(dev(w), 8, 4, rate=rate).cpu().numpy().view(np.uint64)
    assert np.array_equal(tm, oracle.prune_bp_global(w, Mb=8, Nb=4, n_keep=int(np.floor(G / rate + 0.5))))


@pytest.mark.parametrize("Bo,Bi,kr,kc", [(64, 64, 64, 64), (1, 64, 1, 33), (64, 1, 31, 1), (40, 64, 0, 17), (33, 7, 32, 7)])
def test_pack_bb_and_pruning_at_the_edges(Bo, Bi, kr, kc):
    O, I = 2 * Bo, 3 * Bi
    rng = inputs.rng_for(1003)
    w = rng.standard_normal((O, I), dtype=np.float32)
    w[:, 0] = w[:, I - 1]
    rk, ck = npas.prune_bb_magnitude(dev(w), Bo, Bi, kr, kc)
    rk0, ck0 = oracle.prune_bb(w, Bo=Bo, Bi=Bi, keep_rows=kr, keep_cols=kc)
    assert np.array_equal(npas.mask_to_numpy(rk), rk0) and np.array_equal(npas.mask_to_numpy(ck), ck0)
    for dtype in ("f32", "bf16"):
        blob = npas.pack_bb(dev(w), rk, ck, Bo, Bi, torch.float32 if dtype == "f32" else torch.bfloat16)
        assert np.array_equal(blob.data.cpu().numpy(), oracle.pack_bb(w, rk0, ck0, Bo, Bi, dtype))
        wd, r2, c2 = npas.unpack_bb(blob)
        assert torch.equal(wd.float(), torch.from_numpy(oracle.bb_element_mask(rk0, ck0, O, I, Bo, Bi) * w).cuda().to(wd.dtype).float())


def test_masks_that_change_while_they_are_packed():
    """Another stream rewrites the caller's masks all the time, from nothing kept to everything and back: every blob is whole, its
    size, its header and its sections being those of one state of the masks (each word's own)."""
    stop, side = threading.Event(), torch.cuda.Stream()
    rng = inputs.rng_for(1004)
    w = dev(rng.standard_normal((64, 3, 3, 64), dtype=np.float32), "bf16")
    tm = torch.zeros((4, 8), dtype=torch.int64, device="cuda")
    m = dev(rng.standard_normal((128, 192), dtype=np.float32), "bf16")
    both = torch.zeros((2, 2, 3), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()

    def flip():
        with torch.cuda.stream(side):
            while not stop.is_set():
                for v in (-1, 0, 0x155):
                    tm.fill_(v)
                    both.fill_(v)
                side.synchronize()

    t = threading.Thread(target=flip)
    t.start()
    try:
        for _ in range(300):
            blob = npas.pack_bp(w, tm, 16, 8)
            npas.blob_check(blob)
            wd, masks = npas.unpack_bp(blob)
            assert blob.data[:128].view(torch.int32)[15].item() == blob.data.numel()
            words = npas.mask_to_numpy(masks)
            assert set(words.ravel().tolist()) <= {0x1FF, 0, 0x155}
            kept = torch.from_numpy(oracle.bp_element_mask(words, 64, 64, 3, 3, 16, 8)).cuda()
            assert torch.equal(wd, torch.where(kept.bool(), w, torch.zeros_like(w)))
            blob = npas.pack_bb(m, both[0], both[1], 64, 64)
            npas.blob_check(blob)
            assert blob.data[:128].view(torch.int32)[15].item() == blob.data.numel()
            wd, rk, ck = npas.unpack_bb(blob)
            em = oracle.bb_element_mask(npas.mask_to_numpy(rk), npas.mask_to_numpy(ck), 128, 192, 64, 64)
            assert torch.equal(wd, torch.where(torch.from_numpy(em).cuda().bool(), m, torch.zeros_like(m)))
    finally:
        stop.set()
        t.join()
