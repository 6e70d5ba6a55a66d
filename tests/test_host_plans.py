"""What the host chooses before it launches: rules that need no device."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_08923_b200 import binding

N_SMS = 148
SHAPES = {  # d_model, query heads, KV heads, head_dim, d_ffn
    "tiny": (256, 4, 2, 64, 704), "1.5b": (1536, 12, 2, 128, 8960), "8b": (4096, 32, 8, 128, 12288),
}


def _cfg(model, **over):
    d, hq, hkv, hd, f = SHAPES[model]
    base = dict(n_layers=2, d_model=d, n_q_heads=hq, n_kv_heads=hkv, head_dim=hd, d_ffn=f, vocab=1024, tie_lm_head=1, rms_eps=1e-6, rope_theta=1e4,
                mask_token_id=1023, k_max=16, max_batch=64, max_seq_len=4096, page_size=64, beta=1.0, temperature=0.0, sample_seed=0, debug=0, impl=0,
                prefill_rows=4352)
    base.update(over)
    return binding.tidar_config(**base)


def _projections(model):
    d, hq, hkv, hd, f = SHAPES[model]
    return [(0, (hq + 2 * hkv) * hd, d), (0, d, hq * hd), (0, d, f), (1, 2 * f, d)]


@pytest.mark.parametrize("model", list(SHAPES))
def test_epilogues_are_walked_through_only_ahead_of_a_workers_single_item(model):
    lib, out, seen = binding.load(), np.zeros(5, dtype=np.int32), set()
    for R in (1, 20, 96, 97, 272, 288, 289, 600, 1152, 1400, 1776, 2047, 4112):
        for swiglu, N, K in _projections(model):
            assert lib.tidar_debug_plan_projection(C.byref(_cfg(model)), N_SMS, swiglu, R, N, K, binding._ip(out)) == 0
            n_rb, rb_rows, S, items, walked = out.tolist()
            small = R <= 96 or (not swiglu and R <= 288 and N * K <= 15_000_000)
            assert n_rb * rb_rows >= R and 1 <= S <= 8
            if not swiglu:
                assert bool(walked) == (items <= (N_SMS if small else N_SMS // 2)), (R, N, K, out)
                seen.add(walked)
    assert seen == {0, 1} or model == "tiny"
    assert lib.tidar_debug_plan_projection(None, N_SMS, 0, 1, 64, 64, binding._ip(out)) == -1
    assert lib.tidar_debug_plan_projection(C.byref(_cfg(model)), 0, 0, 1, 64, 64, binding._ip(out)) == -1


@pytest.mark.parametrize("n_sms", [148, 144, 143, 132, 100, 96, 74])
def test_bulk_norm_fits_the_shared_memory_it_is_given(n_sms):
    """Every row count and width: the row and its partial results fit the block's shared memory, the blocks of an SM fit beside one another, and on the
    full chip wide rows behind a split projection do go this way."""
    lib, out = binding.load(), np.zeros(2, dtype=np.int32)
    taken = 0
    for R in range(90, 300):
        for d in range(64, 12289, 64):
            for S in (0, 1, 2, 4, 8) if d % 128 == 0 else (3, 4, 5, 6, 7):
                assert lib.tidar_debug_plan_norm(n_sms, R, d, S, binding._ip(out)) == 0
                if out[0]:
                    assert 96 < R <= 288 and 48 * 1024 <= (S + 1) * d * 4 <= out[1], (R, d, S, out)
                    assert -(-R // n_sms) * out[1] <= 200 * 1024
                    taken += 1
    assert taken > 0
    assert lib.tidar_debug_plan_norm(148, 272, 4096, 4, binding._ip(out)) == 0 and out.tolist() == [1, 100 * 1024]
    assert lib.tidar_debug_plan_norm(148, 272, 4096, 9, binding._ip(out)) == -1
