"""asynclm_kv_append_rope against the oracle: V rows and every untouched byte bit-exact; rotated K and Q
rows equal to the fp64 rotation rounded once to bf16, up to a rounding tie here and there (the two sides
evaluate pow / sin / cos with different libraries)."""
import numpy as np
import pytest

from oracle import oracle, rope
from paper_2412_07017_b200 import binding as B
from paper_2412_07017_b200 import workload as W

pytestmark = pytest.mark.gpu


def ulp_diff(a_bits, b_bits):
    """Distance in bf16 steps between two arrays of finite bf16 bit patterns."""
    key = lambda x: np.where(x & 0x8000, 0x8000 - (x & 0x7FFF).astype(np.int32), 0x8000 + (x & 0x7FFF).astype(np.int32))
    return np.abs(key(a_bits) - key(b_bits))


@pytest.mark.parametrize("Hq,Hkv,d,theta", [(32, 8, 128, 500000.0), (8, 2, 64, 10000.0)])
def test_rotated_append(Hq, Hkv, d, theta):
    import torch
    from gpu_util import to_bits, to_dev
    shape = W.Shape(Hq, Hkv, d, 16)
    wl = W.make_single_step("rope", shape, [5, 16, 31, 0, 4000, 70000], [12, 1, 2, 7, 40, 3], seed=31,
                            extra_pages=[0, 1, 0, 2, 1, 0], poison_unused=True)
    st = wl.steps[0]
    pool_dev = to_dev(wl.kv_pool)
    q_dev = to_dev(st.q)
    plan = B.asynclm_plan(shape, wl.num_pages, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices)
    B.asynclm_kv_append_rope(plan, to_dev(st.k_new), to_dev(st.v_new), pool_dev, q_dev, theta)
    torch.cuda.synchronize()
    # oracle: rotate in fp64, round once, then the plain bit-copy append of the rotated rows
    pos = np.concatenate([np.arange(c, c + n) for c, n in zip(st.kv_len_before, st.q_len)])
    rot = lambda bits: W.f32_to_bf16_bits(rope.rotate(W.bf16_bits_to_f64(bits), pos, theta).astype(np.float32))
    k_rot, q_rot = rot(st.k_new), rot(st.q)
    ref_pool = wl.kv_pool.copy()
    oracle.kv_append(ref_pool, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices, k_rot, st.v_new)
    got_pool, got_q = to_bits(pool_dev), to_bits(q_dev)
    assert np.array_equal(got_pool[:, 1], ref_pool[:, 1])                        # V and all untouched V slots: exact
    differs = got_pool[:, 0] != ref_pool[:, 0]
    assert differs.mean() < 1e-4                                                  # untouched K slots are exact too
    assert ulp_diff(got_pool[:, 0][differs], ref_pool[:, 0][differs]).max(initial=0) <= 1
    dq = got_q != q_rot
    assert dq.mean() < 1e-3 and ulp_diff(got_q[dq], q_rot[dq]).max(initial=0) <= 1


@pytest.mark.parametrize("Hq,Hkv,d,rotate_q", [(64, 8, 128, True), (8, 8, 128, False), (1, 1, 64, True), (128, 16, 64, True)])
def test_rotated_append_over_head_counts(Hq, Hkv, d, rotate_q):
    """One CTA rotates all heads of a token: fewer heads than a warp has room for, and more than one pass."""
    import torch
    from gpu_util import to_bits, to_dev
    shape = W.Shape(Hq, Hkv, d, 16)
    wl = W.make_single_step("rope_heads", shape, [0, 131071, 40], [3, 2, 17], seed=32, poison_unused=True)
    st = wl.steps[0]
    pool_dev, q_dev = to_dev(wl.kv_pool), to_dev(st.q)
    plan = B.asynclm_plan(shape, wl.num_pages, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices)
    B.asynclm_kv_append_rope(plan, to_dev(st.k_new), to_dev(st.v_new), pool_dev, q_dev if rotate_q else None, 500000.0)
    torch.cuda.synchronize()
    pos = np.concatenate([np.arange(c, c + n) for c, n in zip(st.kv_len_before, st.q_len)])
    rot = lambda bits: W.f32_to_bf16_bits(rope.rotate(W.bf16_bits_to_f64(bits), pos, 500000.0).astype(np.float32))
    ref_pool = wl.kv_pool.copy()
    oracle.kv_append(ref_pool, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices, rot(st.k_new), st.v_new)
    # the two sides evaluate pow / sin / cos with different libraries: a value on a rounding boundary may go either way
    for got, ref in ((to_bits(pool_dev)[:, 0], ref_pool[:, 0]), (to_bits(q_dev), rot(st.q) if rotate_q else st.q)):
        diff = got != ref
        assert diff.mean() < 1e-3 and ulp_diff(got[diff], ref[diff]).max(initial=0) <= 1
    assert np.array_equal(to_bits(pool_dev)[:, 1], ref_pool[:, 1])


@pytest.mark.parametrize("q_lens", [[2000, 1, 367], [2000, 1, 368]])      # 592 CTAs of four tokens, 593
def test_rotated_append_on_both_sides_of_a_wave(q_lens):
    """A launch of about one wave evaluates the angles before it waits for the kernel in front, a longer one requests its rows first."""
    import torch
    from gpu_util import to_bits, to_dev
    shape = W.Shape(2, 1, 64, 16)
    wl = W.make_single_step("rope_waves", shape, [0, 900, 31], q_lens, seed=33, poison_unused=True)
    st = wl.steps[0]
    pool_dev, q_dev = to_dev(wl.kv_pool), to_dev(st.q)
    plan = B.asynclm_plan(shape, wl.num_pages, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices)
    B.asynclm_kv_append_rope(plan, to_dev(st.k_new), to_dev(st.v_new), pool_dev, q_dev, 10000.0)
    torch.cuda.synchronize()
    pos = np.concatenate([np.arange(c, c + n) for c, n in zip(st.kv_len_before, st.q_len)])
    rot = lambda bits: W.f32_to_bf16_bits(rope.rotate(W.bf16_bits_to_f64(bits), pos, 10000.0).astype(np.float32))
    ref_pool = wl.kv_pool.copy()
    oracle.kv_append(ref_pool, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices, rot(st.k_new), st.v_new)
    # (ties of the two sides' sines and cosines, as above)
    for got, ref in ((to_bits(pool_dev)[:, 0], ref_pool[:, 0]), (to_bits(q_dev), rot(st.q))):
        diff = got != ref
        assert diff.mean() < 1e-3 and ulp_diff(got[diff], ref[diff]).max(initial=0) <= 1
    assert np.array_equal(to_bits(pool_dev)[:, 1], ref_pool[:, 1])


# tokens of a CTA: 1, 1, 2, 7, 20, and 4 in several waves; with more heads 2, 4, and 8 in several waves
@pytest.mark.parametrize("tokens,Hq,Hkv", [(444, 2, 1), (445, 2, 1), (593, 2, 1), (3001, 2, 1), (8437, 2, 1), (8881, 2, 1), (9001, 2, 1),
                                           (445, 64, 8), (1775, 64, 8), (8881, 8, 8)])
def test_rotated_append_over_tokens_of_a_cta(tokens, Hq, Hkv):
    """The tokens of a CTA follow from the waves that they make (see test_rope_grid.py): one, a few, the most, with a remainder in the last CTA,
    and grids of more than one wave."""
    import torch
    from gpu_util import to_bits, to_dev
    shape = W.Shape(Hq, Hkv, 64, 16)
    wl = W.make_single_step("rope_tokens", shape, [3, 900, 31], [tokens - 40, 1, 39], seed=34, poison_unused=True)
    st = wl.steps[0]
    pool_dev, q_dev = to_dev(wl.kv_pool), to_dev(st.q)
    plan = B.asynclm_plan(shape, wl.num_pages, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices)
    B.asynclm_kv_append_rope(plan, to_dev(st.k_new), to_dev(st.v_new), pool_dev, q_dev, 10000.0)
    torch.cuda.synchronize()
    pos = np.concatenate([np.arange(c, c + n) for c, n in zip(st.kv_len_before, st.q_len)])
    rot = lambda bits: W.f32_to_bf16_bits(rope.rotate(W.bf16_bits_to_f64(bits), pos, 10000.0).astype(np.float32))
    ref_pool = wl.kv_pool.copy()
    oracle.kv_append(ref_pool, st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices, rot(st.k_new), st.v_new)
    for got, ref in ((to_bits(pool_dev)[:, 0], ref_pool[:, 0]), (to_bits(q_dev), rot(st.q))):
        diff = got != ref
        assert diff.mean() < 1e-3 and ulp_diff(got[diff], ref[diff]).max(initial=0) <= 1
    assert np.array_equal(to_bits(pool_dev)[:, 1], ref_pool[:, 1])
