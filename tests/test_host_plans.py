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
def test_epilogues_are_walked_through_only_ahead_of_a_workers_single_long_item(model):
    lib, out, seen = binding.load(), np.zeros(5, dtype=np.int32), set()
    for R in (1, 20, 96, 97, 272, 288, 289, 600, 1152, 1400, 1776, 2047, 4112):
        for swiglu, N, K in _projections(model):
            assert lib.tidar_debug_plan_projection(C.byref(_cfg(model)), N_SMS, swiglu, R, N, K, binding._ip(out)) == 0
            n_rb, rb_rows, S, items, walked = out.tolist()
            small = R <= 96 or (not swiglu and R <= 288 and N * K <= 15_000_000)
            assert n_rb * rb_rows >= R and 1 <= S <= 8
            if not swiglu:
                if small:
                    continue                             # (their epilogue is never walked through)
                loop = -(-(K // 64) // S) * (2.15 * rb_rows + 50) / 1750          # us
                assert abs(loop - 4) < 1e-3 or bool(walked) == (items <= N_SMS // 2 and loop > 4), (R, N, K, out)
                seen.add(walked)
    assert seen == ({0} if model == "tiny" else {0, 1})
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


def _step_route(model, n, ks, ar, max_clusters):
    """(route, lead of the best time over the best of another route): every page counted slot by slot, every limit in 64 bits."""
    d, hq, hkv, hd, f = SHAPES[model]
    spt = 128 // (hq // hkv)
    units, tiles = [], []                                # (pages, two tiles)
    for m, k in zip(n, ks):
        slots = [(m + 1, None)] if ar else [(m + j + 1, None) for j in range(k)] + [(m + b + 1, b) for b in range(k) for _ in range(k)]

        def pages(part):
            blocks = [b for _, b in part if b is not None]
            return -(-max(v for v, _ in part) // 64) + (-(-(max(blocks) - min(blocks) + 1) * k // 64) if blocks else 0)
        for r in range(0, len(slots), 2 * spt):
            a, b = slots[r:r + spt], slots[r + spt:r + 2 * spt]
            units.append((pages(a + b), bool(b)))
            tiles += [(pages(x), False) for x in (a, b) if x]
    most_items = N_SMS // hkv if len(units) * hkv <= N_SMS else 2 * N_SMS // hkv if 2 * len(units) * hkv < 3 * N_SMS else len(units)
    if len(units) > 256 or most_items <= len(units):
        return (1, 1), 1.0
    times = {}
    for paired, ents in ((True, units), (False, tiles)):
        us = [p * (1.05 if two else 0.56) for p, two in ents]
        for i in range(0, 32, 2):
            limit = max(max(us) / (1 + 0.5 * i), 0.1) * 1.0001
            cut = [min(int(np.ceil(u / limit)), p) for u, (p, _) in zip(us, ents)]
            if sum(cut) > most_items or max(cut) > (32 if max(n) > 768 else 1):
                continue
            store = [(2.5 if two else 1.5) if c > 1 else 0.0 for c, (_, two) in zip(cut, ents)]
            longest = max(u / c + (0.28 if c > 1 else 0.0) + s + 5 for u, c, s in zip(us, cut, store))
            t = longest
            if sum(cut) * hkv > N_SMS:
                t = max(t, hkv * sum(u + c * (5 + s) for u, c, s in zip(us, cut, store)) / N_SMS + 0.5 * longest)
            if sum(cut) > len(cut):
                t += 3 + 0.3 * sum(cut) / len(cut)
            split = int(sum(cut) > len(cut) or (not paired and 2 * len(units) * hkv > N_SMS))
            times.setdefault((1, split), []).append(t)
    best = {r: min(t) for r, t in times.items()}
    ranked = sorted(best.items(), key=lambda x: x[1])
    lead = ranked[1][1] - ranked[0][1] if len(ranked) > 1 else 1.0
    route, t = ranked[0] if ranked else ((1, 1), 1e30)
    t += 1.5 * route[1]
    places = 2 * (-(-len(units) // 4) * 4) if len(set(ks)) > 1 else len(tiles)
    for size, room in zip((2, 4, 8), max_clusters):
        if size * 16 <= hd:
            tc = -(-max(p for p, _ in tiles) // size) * 0.56 + 7
            if places * hkv <= room and 4 * places * hkv * size <= 3 * N_SMS:
                lead = min(lead, abs(tc - (t - 0.3)))
                if tc < t - 0.3:
                    t, route = tc, (size, 0)
    return route, lead


@pytest.mark.parametrize("model", list(SHAPES))
def test_step_attention_follows_the_plan_kernels_estimate(model):
    """Cut, uncut or shared by clusters: random batches, one row and k (k + 1) rows per sequence, equal and mixed block lengths, lengths up to 30 k.
    (Where two routes are within a thousandth of a microsecond, 32-bit sums may choose either.)"""
    lib, out, rng, seen = binding.load(), np.zeros(2, dtype=np.int32), np.random.default_rng(5), {}
    room = np.array([74, 36, 16], dtype=np.int32)
    for i in range(250):
        ar, mixed = i % 4 == 0, i % 4 == 1
        n_seqs = int(rng.integers(1, 41 if ar else 5))
        n = rng.integers(0, int(np.exp(rng.uniform(np.log(20), np.log(30000)))), n_seqs).astype(np.int32)
        k = 1 if ar else int(rng.integers(1, 17))
        ks = (rng.integers(1, k + 1, n_seqs) if mixed else np.full(n_seqs, k)).astype(np.int32)
        assert lib.tidar_debug_plan_step(C.byref(_cfg(model)), N_SMS, binding._ip(room), binding._ip(n), binding._ip(ks), n_seqs, int(ar), binding._ip(out)) == 0
        route, lead = _step_route(model, n.tolist(), ks.tolist(), ar, room.tolist())
        assert lead < 1e-3 or tuple(out.tolist()) == route, (n, ks, ar, out, route)
        seen[route] = seen.get(route, 0) + 1
    assert len(seen) >= 4 and (1, 0) in seen and (1, 1) in seen, seen
