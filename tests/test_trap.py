"""Trap handler (paper Section 5.4): the library's decision rule and swap kernels against the oracle."""
import numpy as np
import pytest

from oracle import trap
from paper_2412_07017_b200 import binding as B
from paper_2412_07017_b200 import workload as W


def test_decision_rule_matches_the_oracle_on_a_grid():
    g = np.random.default_rng(0)
    for _ in range(20):
        m = dict(swap_fixed_us=g.uniform(0, 500), swap_us_per_token=g.uniform(0.1, 100),
                 recompute_fixed_us=g.uniform(0, 5000), recompute_us_per_token=g.uniform(0, 100),
                 recompute_us_per_token2=g.uniform(0, 0.2))
        for n in (0, 1, 17, 300, 4096, 100000):
            for w in (0.0, 10.0, 1e3, 1e5, 1e9):
                dec, s, r = B.asynclm_trap_decide(m, n, w)
                assert dec == trap.decide(m, n, w)
                assert s == pytest.approx(trap.swap_us(m, n)) and r == pytest.approx(trap.recompute_us(m, n))
    assert (B.TRAP_KEEP, B.TRAP_SWAP, B.TRAP_RECOMPUTE) == (trap.KEEP, trap.SWAP, trap.RECOMPUTE)


def test_swap_argument_checks_need_no_gpu():
    import ctypes
    lib = B.load()
    cs = B._cshape(W.Shape(8, 2, 64, 16), 10)
    ids = np.array([1, 2, 12], dtype=np.int32)
    buf = np.zeros(1 << 16, dtype=np.uint8)
    a = buf.ctypes.data + (-buf.ctypes.data % 256)
    assert lib.asynclm_kv_swap_out(ctypes.byref(cs), ids.ctypes.data, 3, a, a, a, None) == -3      # id outside the pool
    ids[2] = 2
    assert lib.asynclm_kv_swap_in(ctypes.byref(cs), ids.ctypes.data, 3, a, a, a, None) == -3       # duplicate destination
    assert lib.asynclm_kv_swap_in(ctypes.byref(cs), ids.ctypes.data, 3, a, a + 8, a, None) == -1   # misaligned
    assert lib.asynclm_kv_swap_out(ctypes.byref(cs), None, 0, None, None, None, None) == 0
    assert B.kv_swap_staging_bytes(W.Shape(8, 2, 64, 16), 10, 3) >= 3 * 2 * 2 * 16 * 64 * 2 + 12


@pytest.mark.gpu
@pytest.mark.parametrize("Hq,Hkv,d", [(32, 8, 128), (8, 2, 64)])
def test_swap_out_and_in_are_bit_copies(Hq, Hkv, d):
    """A paused sequence's pages go to pinned host memory and come back into other pages: the image,
    the pool after the swap-in and every untouched page agree with the oracle byte for byte."""
    import torch
    from gpu_util import to_bits, to_dev
    shape = W.Shape(Hq, Hkv, d, 16)
    wl = W.make_single_step("swap", shape, [700, 333, 90], [1, 0, 1], seed=21, spare_pages=60)
    st = wl.steps[0]
    pool_dev = to_dev(wl.kv_pool)
    ref_pool = wl.kv_pool.copy()
    b = 1                                                     # the paused sequence
    old = st.page_indices[st.page_indptr[b]:st.page_indptr[b + 1]]
    n = len(old)
    staging = torch.empty(B.kv_swap_staging_bytes(shape, wl.num_pages, n), dtype=torch.uint8, device="cuda")
    image = torch.zeros((n,) + wl.kv_pool.shape[1:], dtype=torch.int16).pin_memory()
    B.asynclm_kv_swap_out(shape, wl.num_pages, old, pool_dev, staging, image)
    torch.cuda.synchronize()
    ref_image = trap.swap_out(ref_pool, old)
    assert np.array_equal(image.numpy().view(np.uint16), ref_image)
    assert np.array_equal(to_bits(pool_dev), ref_pool)                      # swap-out does not write the pool
    # the old pages are reused by someone else, the sequence comes back into pages nobody owns
    pool_dev[torch.from_numpy(old.astype(np.int64)).cuda()] = 0
    ref_pool[old] = 0
    used = set(st.page_indices.tolist())
    new = np.array([p for p in np.random.default_rng(3).permutation(wl.num_pages) if p not in used][:n], dtype=np.int32)
    B.asynclm_kv_swap_in(shape, wl.num_pages, new, pool_dev, staging, image)
    torch.cuda.synchronize()
    trap.swap_in(ref_pool, new, ref_image)
    assert np.array_equal(to_bits(pool_dev), ref_pool)


@pytest.mark.gpu
@pytest.mark.parametrize("hk,pages,memory", [(1, 1, "pinned"), (1, 511, "pinned"), (1, 512, "pinned"), (1, 513, "pinned"),
                                             (1, 960, "pinned"), (1, 961, "pinned"), (3, 170, "pinned"), (3, 171, "pinned"),
                                             (1, 300, "pinned"), (1, 512, "pageable"), (1, 961, "pageable"), (1, 300, "captured")])
def test_swaps_in_place_and_through_staging(hk, pages, memory):
    """Images up to and beyond 2 MB (4096 bytes a page and head) and page ids up to and beyond those that parameters hold, behind
    one another in one stream.  What is left in the staging buffer says which way they went: nothing of a swap in place, the image of
    the others, and behind it the ids where they were copied."""
    import torch
    shape, num = W.Shape(8, hk, 64, 16), 1200
    g = np.random.default_rng(pages)
    pool = g.integers(0, 1 << 16, (num, 2, hk, 16, 64)).astype(np.uint16)
    old, new = (g.permutation(num)[:pages].astype(np.int32) for _ in range(2))
    want_image = trap.swap_out(pool, old)
    want = np.zeros_like(pool)
    trap.swap_in(want, new, want_image)
    src, dst = torch.from_numpy(pool.view(np.int16)).cuda(), torch.zeros(pool.shape, dtype=torch.int16, device="cuda")
    staging = torch.empty(B.kv_swap_staging_bytes(shape, num, pages), dtype=torch.uint8, device="cuda")
    staging.fill_(0xA5)
    whole = torch.full((pages + 2,) + pool.shape[1:], 77, dtype=torch.int16)
    whole = whole if memory == "pageable" else whole.pin_memory()
    image = whole[1:-1]
    out = lambda ids: B.asynclm_kv_swap_out(shape, num, ids, src, staging, image)
    back = lambda ids: B.asynclm_kv_swap_in(shape, num, ids, dst, staging, image)
    torch.cuda.synchronize()
    if memory == "captured":      # the graph reads ids and image when it runs
        ids = torch.empty((2, pages), dtype=torch.int32).pin_memory()
        ids[:] = torch.arange(pages, dtype=torch.int32)
        graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=s):
            out(ids[0].numpy()), back(ids[1].numpy())
        ids[0], ids[1] = torch.from_numpy(old), torch.from_numpy(new)
        graph.replay()
    else:
        for k in range(3):
            ids = old.copy()
            out(ids)
            ids[:] = 0
            if memory == "pageable":
                torch.cuda.synchronize()
            ids = new.copy()
            back(ids)
            ids[:] = 0
    torch.cuda.synchronize()
    assert np.array_equal(image.numpy().view(np.uint16), want_image) and (whole[0] == 77).all() and (whole[-1] == 77).all()
    assert np.array_equal(dst.cpu().numpy().view(np.uint16), want) and np.array_equal(src.cpu().numpy().view(np.uint16), pool)
    used = staging.cpu().numpy()
    image_bytes = want_image.nbytes
    in_place = memory == "pinned" and image_bytes <= 2 << 20
    ids_copied = memory == "captured" or pages > 960
    assert (used[:image_bytes] == 0xA5).all() if in_place else np.array_equal(used[:image_bytes].view(np.uint16), want_image.reshape(-1))
    assert np.array_equal(used[image_bytes:image_bytes + 4 * pages].view(np.int32), new) if ids_copied else (used[image_bytes:] == 0xA5).all()


@pytest.mark.gpu
def test_an_image_in_two_registrations_is_refused():
    """Page-locked in two parts that no single range covers: no kernel touches it, and the copy refuses it."""
    import torch
    shape, num, pages = W.Shape(8, 1, 64, 16), 200, 100
    pool = torch.ones((num, 2, 1, 16, 64), dtype=torch.int16, device="cuda")
    staging = torch.zeros(B.kv_swap_staging_bytes(shape, num, pages), dtype=torch.uint8, device="cuda")
    base = torch.zeros(pages * 4096 + 8192, dtype=torch.uint8)
    base, rt = base[-base.data_ptr() % 4096:], torch.cuda.cudart()
    image, ids, cut = base[:pages * 4096], np.arange(pages, dtype=np.int32), 32768
    parts = [(image.data_ptr(), cut), (image.data_ptr() + cut, pages * 4096 - cut)]
    torch.cuda.synchronize()
    for p, n in parts:
        assert int(rt.cudaHostRegister(p, n, 0)) == 0
    try:
        for call in (B.asynclm_kv_swap_out, B.asynclm_kv_swap_in):
            with pytest.raises(B.AsynclmError, match="CUDA"):
                call(shape, num, ids, pool, staging, image)
        torch.cuda.synchronize()
    finally:
        for p, n in parts:
            rt.cudaHostUnregister(p)
    assert not image.any() and (pool == 1).all()
