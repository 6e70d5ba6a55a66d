"""Structured-mask paged attention alone vs the oracle's dense-mask attention (needs a B200)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import tidar_oracle as O
from tests.helpers import make_model
from tidar_synth import CONFIGS, gen_normal_bf16, tensor_id

pytestmark = pytest.mark.gpu

IMPLS = [0, 1]
TOL = 3e-2          # unit-variance bf16 inputs; bf16 output rounding alone is ~1e-2 at |x| ~ 3


def _ctx(hd, Hq, Hkv, k_max, max_batch, impl):
    from paper_2511_08923_b200 import Tidar, pack_weights
    sh = replace(CONFIGS["tiny"], head_dim=hd, n_q_heads=Hq, n_kv_heads=Hkv, n_layers=1, vocab=64, d_ffn=64, d_model=64)
    from tidar_synth import gen_model_weights
    return Tidar(sh, pack_weights(gen_model_weights(sh), "cuda:0"), k_max=k_max, max_batch=max_batch, max_seq_len=128,
                 impl=impl)


def _case(t, hd, Hq, Hkv, k, ns, seed):
    B, T, page = len(ns), k * (k + 1), 64
    pps = (max(ns) + k + page - 1) // page
    n_pages = B * pps + 3
    dev = "cuda:0"
    q = gen_normal_bf16(seed, tensor_id("q"), B * T * Hq * hd, 1.0).view(B * T, Hq, hd)
    kl = gen_normal_bf16(seed, tensor_id("k", 1), B * k * k * Hkv * hd, 1.0).view(B * k * k, Hkv, hd)
    vl = gen_normal_bf16(seed, tensor_id("v", 1), B * k * k * Hkv * hd, 1.0).view(B * k * k, Hkv, hd)
    kp = torch.zeros(n_pages, Hkv, page, hd, dtype=torch.bfloat16)
    vp = torch.zeros(n_pages, Hkv, page, hd, dtype=torch.bfloat16)
    perm = torch.randperm(n_pages, generator=torch.Generator().manual_seed(seed))
    pt = perm[:B * pps].view(B, pps).to(torch.int32)
    refs = []
    for s, n in enumerate(ns):
        kc = gen_normal_bf16(seed, tensor_id("k", 2 + s), (n + k) * Hkv * hd, 1.0).view(n + k, Hkv, hd)
        vc = gen_normal_bf16(seed, tensor_id("v", 2 + s), (n + k) * Hkv * hd, 1.0).view(n + k, Hkv, hd)
        for p in range(n + k):
            kp[pt[s, p // page], :, p % page] = kc[p]
            vp[pt[s, p // page], :, p % page] = vc[p]
        k_all = torch.cat([kc, kl[s * k * k:(s + 1) * k * k]]).double().numpy()
        v_all = torch.cat([vc, vl[s * k * k:(s + 1) * k * k]]).double().numpy()
        refs.append(O.masked_attention(q[s * T:(s + 1) * T].double().numpy(), k_all, v_all, O.build_decode_mask(n, k)))
    out = torch.full((B * T, Hq * hd), float("nan"), dtype=torch.bfloat16, device=dev)
    sl = torch.tensor(ns, dtype=torch.int32, device=dev)
    t.attention(q.to(dev), kp.to(dev), vp.to(dev), pt.to(dev), sl, kl.to(dev), vl.to(dev), out, B, k)
    torch.cuda.synchronize()
    got = out.float().cpu().numpy().reshape(B * T, Hq, hd)
    ref = np.concatenate(refs)
    assert np.isfinite(got).all()
    assert np.abs(got - ref).max() <= TOL


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("hd,Hq,Hkv", [(64, 4, 2), (128, 8, 2), (128, 4, 4)])
def test_attention_small_lengths(impl, hd, Hq, Hkv):
    t = _ctx(hd, Hq, Hkv, 8, 3, impl)
    # prefix lengths around page boundaries, n = 0 included (first token of a sequence)
    _case(t, hd, Hq, Hkv, 4, [0, 1, 63], 11)
    _case(t, hd, Hq, Hkv, 4, [64, 65, 127], 12)
    _case(t, hd, Hq, Hkv, 8, [200, 5], 13)
    _case(t, hd, Hq, Hkv, 1, [9], 14)
    _case(t, hd, Hq, Hkv, 3, [700], 15)
    t.close()


@pytest.mark.parametrize("impl", IMPLS)
def test_attention_k16_long_prefix(impl):
    t = _ctx(128, 8, 2, 16, 1, impl)
    _case(t, 128, 8, 2, 16, [1500], 21)
    t.close()


def _case_sampled(t, hd, Hq, Hkv, k, n, seed, n_rows=24):
    """Config-2 sizes: the kernel runs on all rows, the oracle on a sample of query rows
    (each with its own dense-mask row), which covers every kind of slot and both ends."""
    T, page = k * (k + 1), 64
    pps = (n + k + page - 1) // page
    dev = "cuda:0"
    q = gen_normal_bf16(seed, tensor_id("q"), T * Hq * hd, 1.0).view(T, Hq, hd)
    kl = gen_normal_bf16(seed, tensor_id("k", 1), k * k * Hkv * hd, 1.0).view(k * k, Hkv, hd)
    vl = gen_normal_bf16(seed, tensor_id("v", 1), k * k * Hkv * hd, 1.0).view(k * k, Hkv, hd)
    kc = gen_normal_bf16(seed, tensor_id("k", 2), pps * page * Hkv * hd, 1.0).view(pps * page, Hkv, hd)
    vc = gen_normal_bf16(seed, tensor_id("v", 2), pps * page * Hkv * hd, 1.0).view(pps * page, Hkv, hd)
    perm = torch.randperm(pps + 5, generator=torch.Generator().manual_seed(seed))[:pps]
    kp = torch.zeros(pps + 5, Hkv, page, hd, dtype=torch.bfloat16)
    vp = torch.zeros(pps + 5, Hkv, page, hd, dtype=torch.bfloat16)
    kp[perm] = kc.view(pps, page, Hkv, hd).permute(0, 2, 1, 3)
    vp[perm] = vc.view(pps, page, Hkv, hd).permute(0, 2, 1, 3)
    out = torch.full((T, Hq * hd), float("nan"), dtype=torch.bfloat16, device=dev)
    t.attention(q.to(dev), kp.to(dev), vp.to(dev), perm.view(1, pps).to(torch.int32).to(dev),
                torch.tensor([n], dtype=torch.int32, device=dev), kl.to(dev), vl.to(dev), out, 1, k)
    torch.cuda.synchronize()
    got = out.float().cpu().numpy().reshape(T, Hq, hd)
    assert np.isfinite(got).all()
    rows = np.unique(np.concatenate([[0, k - 1, k, T - 1], np.random.default_rng(seed).integers(0, T, n_rows)]))
    mask = O.build_decode_mask(n, k)[rows]
    k_all = torch.cat([kc[:n + k], kl]).double().numpy()
    v_all = torch.cat([vc[:n + k], vl]).double().numpy()
    ref = O.masked_attention(q[rows].double().numpy(), k_all, v_all, mask)
    assert np.abs(got[rows] - ref).max() <= TOL


@pytest.mark.parametrize("n", [1024, 4096, 16384, 32768])
def test_attention_microbench_sizes_sampled_rows(n):
    """32 query / 8 KV heads, head_dim 128, k = 16: the stand-alone attention workload."""
    from paper_2511_08923_b200 import Tidar, pack_weights
    from tidar_synth import gen_model_weights
    sh = replace(CONFIGS["tiny"], head_dim=128, n_q_heads=32, n_kv_heads=8, n_layers=1, vocab=64, d_ffn=64, d_model=64)
    t = Tidar(sh, pack_weights(gen_model_weights(sh), "cuda:0"), k_max=16, max_batch=1, max_seq_len=128, impl=0)
    _case_sampled(t, 128, 32, 8, 16, n, 40 + n % 97)
    t.close()


@pytest.mark.parametrize("ns,k", [
    ([3000, 5, 700], 4),          # one long sequence among short ones: its key range is cut into items, the others' are not
    ([2500], 1),                  # a single query tile: more items than the page ids one warp holds at a time
    ([2] * 200 + [300] * 30, 1),  # more (tile pair, KV head) units than three for two SMs: nothing is split
    ([1, 0, 66] * 180, 1),        # more tile pairs than the plan ranks by length
])
def test_attention_work_plan(ns, k):
    t = _ctx(64, 4, 2, 8, 32, 0)
    _case(t, 64, 4, 2, k, ns, 31)
    cluster, merge, cut = t.attention_route()
    assert cluster == 1 and (not merge or cut != 0)              # (a merge kernel comes with key ranges that were cut)
    t.close()


@pytest.mark.parametrize("hd,Hq,Hkv,k,ns,launches", [
    # one kernel, two streams per tile; from 16 pages on key ranges are cut and a merge kernel follows, the same number of items for every
    # tile; with too few SMs for that the call is planned
    (128, 8, 2, 1, [15 * 64 - 1], 1), (128, 8, 2, 1, [15 * 64], 2), (64, 4, 2, 12, [5000], 2),
    (64, 4, 2, 3, [2500, 100, 700, 0, 400], 2),                    # eight items for the first, one or a few for the others
    (128, 32, 8, 16, [1300], 1), (128, 32, 8, 16, [1700], 3),
    (64, 4, 2, 8, [0, 1, 63, 64, 65, 700, 1], 1),
    (128, 12, 2, 5, [300, 62, 63], 1),                             # 21 slots per tile: two unused rows
    # one stream per tile, two CTAs per SM: between one and two tiles per SM
    (128, 32, 8, 16, [0, 63, 64, 700], 1),                         # 288 tiles, the last of a sequence half empty
    (64, 4, 2, 8, [(37 * i) % 300 for i in range(49)] + [2000], 1),
    (64, 4, 2, 8, [5] * 49 + [2600], 3),                           # 41 pages: planned
    (128, 12, 2, 5, [(11 * i) % 130 for i in range(40)], 1),
    (128, 8, 8, 2, [1, 70] * 15, 1),                               # one head per KV head: a tile holds whole sequences' slots
])
def test_attention_without_a_plan(hd, Hq, Hkv, k, ns, launches):
    t = _ctx(hd, Hq, Hkv, k, len(ns), 0)
    before = t.launch_count()
    _case(t, hd, Hq, Hkv, k, ns, 51)
    assert t.launch_count() - before == launches
    t.close()


@pytest.mark.parametrize("hd,Hq,Hkv,k,ns,size", [
    (128, 8, 2, 1, [600], 8), (128, 8, 2, 4, [900, 0, 70, 320], 8),       # some tiles are not shared; six pages: CTAs of a sharing cluster without any
    (128, 12, 2, 16, [640], 4), (64, 4, 2, 8, [700, 1, 350, 64], 4),      # two unused rows per tile; head_dim 64
    (128, 32, 8, 16, [1000], 2), (64, 8, 8, 16, [900], 4),                # one head per KV head
    (128, 32, 8, 16, [400], 1), (128, 8, 2, 4, [200], 1),                 # too few pages
])
def test_attention_shared_by_clusters(hd, Hq, Hkv, k, ns, size):
    t = _ctx(hd, Hq, Hkv, k, len(ns), 0)
    before = t.launch_count()
    _case(t, hd, Hq, Hkv, k, ns, 61)
    assert t.launch_count() - before == 1
    assert t.attention_route() == (size, False, -1)
    t.close()


@pytest.mark.parametrize("hd,Hq,Hkv,k,lens", [
    (128, 32, 8, 4, [100]), (128, 32, 8, 16, [100]), (128, 12, 2, 16, [200]), (64, 4, 2, 8, [0, 50, 100, 200]),     # clusters of eight, two, four, eight
])
def test_a_page_table_wider_than_the_lengths_changes_nothing(hd, Hq, Hkv, k, lens):
    """Short sequences under a table wide enough for a call to be launched in clusters: bit for bit what the narrow table gives, for a tile of few pages
    is not shared."""
    dev, b = "cuda:0", len(lens)
    t = _ctx(hd, Hq, Hkv, k, b, 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(k)

    def rnd(*shape):
        return torch.randn(*shape, device=dev, dtype=torch.bfloat16, generator=gen)
    T, W = k * (k + 1), 12
    q, kp, vp, kl, vl = rnd(b * T, Hq, hd), rnd(b * W, Hkv, 64, hd), rnd(b * W, Hkv, 64, hd), rnd(b * k * k, Hkv, hd), rnd(b * k * k, Hkv, hd)
    table = torch.randperm(b * W, device=dev, generator=gen).to(torch.int32).view(b, W)
    outs = []
    for width in (4, W):
        out = torch.full((b * T, Hq * hd), float("nan"), dtype=torch.bfloat16, device=dev)
        t.attention(q, kp, vp, table[:, :width].contiguous(), torch.tensor(lens, dtype=torch.int32, device=dev), kl, vl, out, b, k)
        t.sync()
        outs.append(out)
    assert torch.isfinite(outs[0]).all() and torch.equal(outs[0], outs[1])
    t.close()


def test_attention_clamps_lengths_and_page_indices_without_a_plan():
    """Lengths below 0 and beyond the table's positions are clamped on every route, and a page outside the pool reads as zeros: both the
    two-stream and the one-stream instance against the same call with legal values."""
    hd, Hq, Hkv, k, dev = 64, 4, 2, 8, "cuda:0"
    for b in (2, 50):
        t = _ctx(hd, Hq, Hkv, k, b, 0)
        gen = torch.Generator(device=dev)
        gen.manual_seed(b)

        def rnd(*shape):
            return torch.randn(*shape, device=dev, dtype=torch.bfloat16, generator=gen)
        q, kp, vp, kl, vl = rnd(b * 72, Hq, hd), rnd(2 * b + 1, Hkv, 64, hd), rnd(2 * b + 1, Hkv, 64, hd), rnd(b * 64, Hkv, hd), rnd(b * 64, Hkv, hd)
        kp[2 * b], vp[2 * b] = 0, 0
        legal = torch.arange(2 * b, dtype=torch.int32, device=dev).view(b, 2)
        legal[1, 0] = 2 * b
        wild = legal.clone()
        wild[1, 0] = 1 << 20
        outs = []
        for table, lens in ((legal, [0, 120] * (b // 2)), (wild, [-5, 100000] * (b // 2))):
            out = torch.full((b * 72, Hq * hd), float("nan"), dtype=torch.bfloat16, device=dev)
            before = t.launch_count()
            t.attention(q, kp, vp, table, torch.tensor(lens, dtype=torch.int32, device=dev), kl, vl, out, b, k)
            t.sync()
            assert t.launch_count() - before == 1
            outs.append(out)
        assert torch.isfinite(outs[0]).all() and torch.equal(outs[0], outs[1])
        t.close()


def test_attention_beyond_32767_pages():
    """One sequence of 32770 pages.  Scores are small (weights within e^+-0.4 of each other) and V rises with the position, so that the output
    says which part of the cache was attended to: 0.5 for all of it.  Bound: bf16 rounding of the output, 2^-9 x 0.5, of V (the same,
    averaged over two million positions) and of P (the same): 4e-3 is four times their sum."""
    n, k, hq, hd, dev = 32769 * 64 + 30, 2, 2, 64, "cuda:0"
    pages = (n + k + 63) // 64
    t = _ctx(hd, hq, 1, k, 1, 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(7)

    def rnd(*shape):
        return torch.randn(*shape, device=dev, dtype=torch.bfloat16, generator=gen)
    q, kp = rnd(k * (k + 1), hq, hd) * 0.1, rnd(pages, 1, 64, hd)
    ramp = torch.arange(pages * 64, device=dev, dtype=torch.float32) / n
    vp = ramp.to(torch.bfloat16).view(pages, 1, 64, 1).expand(pages, 1, 64, hd).contiguous()
    kl, vl = rnd(k * k, 1, hd), rnd(k * k, 1, hd)
    table = torch.randperm(pages, device=dev, generator=gen)
    kp2, vp2 = torch.empty_like(kp), torch.empty_like(vp)
    kp2[table], vp2[table] = kp, vp                     # position p lies in page table[p / 64]
    out = torch.full((k * (k + 1), hq * hd), float("nan"), dtype=torch.bfloat16, device=dev)
    t.attention(q, kp2, vp2, table.to(torch.int32).view(1, pages), torch.tensor([n], dtype=torch.int32, device=dev), kl, vl, out, 1, k)
    t.sync()
    got = out.float().view(k * (k + 1), hq, hd)
    keys, vals = kp.view(-1, hd)[:n + k].float(), vp.view(-1, hd)[:n + k, 0].double()
    for r in range(k * (k + 1)):
        b = (r - k) // k
        seen = n + r + 1 if r < k else n + b + 1
        for h in range(hq):
            s = keys[:seen] @ q[r, h].float() / hd ** 0.5
            if r >= k:
                s = torch.cat([s, kl[b * k:(b + 1) * k, 0].float() @ q[r, h].float() / hd ** 0.5])
            w = torch.softmax(s.double(), 0)
            want = w[:seen] @ vals[:seen]
            if r >= k:
                want = want + w[seen:] @ vl[b * k:(b + 1) * k, 0].double()
            assert (got[r, h].double() - want).abs().max() <= 4e-3, (r, h)
    t.close()
