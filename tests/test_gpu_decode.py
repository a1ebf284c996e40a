"""The generation step over a cache (Section 3.1, Eq. 2-3) through the C ABI against the fp64 oracle.

Tolerance: the kernel multiplies bf16 values exactly in fp32, accumulates in fp32 and takes
exponentials with ex2.approx (2 ulp), so every output element carries a few 1e-7 of the sum of
|p_j v_j|; the tests assert |got - ref| <= 1e-3 |ref| + 1e-5 (values are O(1)).  The appended cache
row must equal the new token's row bit for bit and no other cache element may change.
"""
import numpy as np
import pytest

from oracle import lookm_oracle as orc
from paper_2406_18139_b200 import synth
from tests.helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2406_18139_b200 import binding
    binding.lib()
    return binding


def _bits(shape, key, scale=1.0):
    x = synth.normal(synth.stream_key(*key), int(np.prod(shape))).reshape(shape) * scale
    return synth.f32_to_bf16_bits(x.astype(np.float32))


def close(got, ref):
    return np.abs(got - ref) <= 1e-3 * np.abs(ref) + 1e-5


def run_step(B, Hq, Hkv, n, cap, packed, seed, scale=0.0, q_scale=1.0):
    """One request: cache of n rows in a buffer with room for `cap`; returns nothing, asserts."""
    import torch
    ck_b, cv_b = _bits((Hkv, cap, 128), (seed, 1)), _bits((Hkv, cap, 128), (seed, 2))
    q_b, kn_b, vn_b = _bits((Hq, 128), (seed, 3), q_scale), _bits((Hkv, 128), (seed, 4)), _bits((Hkv, 128), (seed, 5))
    if packed:                                            # [rows, Hkv, 128]
        dk, dv = to_dev(ck_b.transpose(1, 0, 2).copy()), to_dev(cv_b.transpose(1, 0, 2).copy())
        lay = B.CacheLayout(Hq, Hkv, 128, Hkv * 128, 128, scale)
    else:                                                 # [Hkv, cap, 128]
        dk, dv = to_dev(ck_b), to_dev(cv_b)
        lay = B.CacheLayout(Hq, Hkv, 128, 128, cap * 128, scale)
    q, kn, vn = to_dev(q_b), to_dev(kn_b), to_dev(vn_b)
    out = torch.full((Hq, 128), np.nan, dtype=torch.float32, device="cuda")
    ws = B.alloc_decode_workspace(lay)
    before_k, before_v = dk.clone(), dv.clone()
    B.check(B.lookm_decode_step(q, kn, vn, dk, dv, n, lay, out, ws))
    torch.cuda.synchronize()
    f = synth.bf16_to_f32
    ref, _, _ = orc.decode_step(f(q_b), f(kn_b), f(vn_b), f(ck_b)[:, :n], f(cv_b)[:, :n],
                                scale=None if scale == 0.0 else scale)
    got = out.cpu().numpy().astype(np.float64)
    assert close(got, ref).all(), float(np.abs(got - ref).max())
    # Eq. 2: row n now holds the new token's rows; everything else is as before
    view = (lambda t: t.transpose(0, 1)) if packed else (lambda t: t)
    assert torch.equal(view(dk)[:, n], kn) and torch.equal(view(dv)[:, n], vn)
    keep = torch.ones(cap, dtype=torch.bool, device="cuda")
    keep[n] = False
    assert torch.equal(view(dk)[:, keep], view(before_k)[:, keep])
    assert torch.equal(view(dv)[:, keep], view(before_v)[:, keep])
    # a second identical step on the same state gives the same bits (fixed order of additions)
    out2 = torch.zeros_like(out)
    B.check(B.lookm_decode_step(q, kn, vn, dk, dv, n, lay, out2, ws))
    torch.cuda.synchronize()
    assert torch.equal(out, out2)


@pytest.mark.parametrize("Hq,Hkv,n,packed", [(1, 1, 0, False), (1, 1, 1, True), (4, 2, 17, False),
                                             (4, 4, 63, True), (8, 1, 64, False), (32, 8, 65, True),
                                             (6, 2, 200, False), (32, 32, 1000, False), (16, 1, 777, True)])
def test_one_step_small_caches(B, Hq, Hkv, n, packed):
    run_step(B, Hq, Hkv, n, n + 3, packed, seed=600 + n)


@pytest.mark.parametrize("Hq,Hkv,n,packed", [(2, 1, 15, False), (3, 1, 16, True), (10, 2, 31, False), (6, 1, 14, True),
                                             (7, 1, 63, False), (16, 2, 128, True), (12, 1, 500, False), (22, 2, 40, False),
                                             (64, 4, 2047, True), (8, 2, 9001, False)])
def test_grouped_queries_at_the_edges_of_sixteen_row_steps(B, Hq, Hkv, n, packed):
    """Groups of 2 to 16 heads (padded to 2, 4 or 8, cut into passes; 11 is prime: one head per pass),
    with the appended row first, last and in the middle of a step, and splits with idle warps."""
    run_step(B, Hq, Hkv, n, n + 2, packed, seed=760 + n, q_scale=1.0 + (n % 3))


@pytest.mark.parametrize("Hq,Hkv,n,q_scale", [(16, 2, 30000, 1.0), (32, 8, 12000, 1.0), (16, 2, 30000, 6.0), (16, 4, 20000, 3.0)])
def test_grouped_queries_are_as_precise_as_single_ones(B, Hq, Hkv, n, q_scale):
    """The same step with the KV heads repeated, so that every query head has rows of its own and everything
    is computed in fp32: the grouped step's error against fp64 may be half as large again (they were equal
    within 20 % over 24 draws each; sums left to the tensor core alone had 1.3 to 2.5 times the error)."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(n + Hq)
    rand = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    g, err = Hq // Hkv, np.zeros(2)
    for _ in range(4):
        k, v, kn, vn = (rand(*s, 128).bfloat16() for s in ((Hkv, n + 1), (Hkv, n + 1), (Hkv,), (Hkv,)))
        q = (rand(Hq, 128) * q_scale).bfloat16()
        k[:, n], v[:, n] = kn, vn
        p = torch.softmax(torch.einsum("hgd,hnd->hgn", q.double().view(Hkv, g, 128), k.double()) * 128 ** -0.5, dim=-1)
        ref = torch.einsum("hgn,hnd->hgd", p, v.double()).view(Hq, 128)
        for i, rep in enumerate((1, g)):
            kk, vv, kkn, vvn = (t.repeat_interleave(rep, dim=0).contiguous() for t in (k, v, kn, vn))
            lay = B.CacheLayout(Hq, Hkv * rep, 128, 128, (n + 1) * 128, 0.0)
            out = torch.zeros(Hq, 128, device="cuda")
            B.check(B.lookm_decode_step(q, kkn, vvn, kk, vv, n, lay, out, B.alloc_decode_workspace(lay)))
            err[i] += float((out.double() - ref).norm() / ref.norm())
    assert err[0] <= 1.5 * err[1], err / 4


@pytest.mark.parametrize("Hq,Hkv,n", [(2, 2, 300), (2, 1, 300), (4, 1, 300), (8, 1, 300), (12, 2, 3000), (4, 2, 9000), (16, 4, 40),
                                      (76, 76, 1600)])
def test_logits_of_minus_infinity_and_infinite_values(B, Hq, Hkv, n):
    """Rows whose logits overflow to -inf count nothing, also where a warp meets them first; an infinite
    value makes its feature infinite and leaves the others alone.  One query head or several per row."""
    import torch
    k, v = (synth.bf16_to_f32(_bits((Hkv, n, 128), (870 + n, i))) for i in (1, 2))
    q = np.abs(synth.bf16_to_f32(_bits((Hq, 128), (870 + n, 3)))) + 1.0
    k[:, :n // 2] = -3e38                                 # q . k = -inf in fp32, a weight of zero either way
    k[:, n // 2 + 5, :] = -3e38
    v[:, n // 2 + 1, 7], v[:, n // 2 + 2, 9] = np.inf, -np.inf
    kn, vn = (synth.bf16_to_f32(_bits((Hkv, 128), (870 + n, i))) for i in (4, 5))
    bits = [synth.f32_to_bf16_bits(np.ascontiguousarray(x)) for x in (q, kn, vn, np.pad(k, ((0, 0), (0, 1), (0, 0))), np.pad(v, ((0, 0), (0, 1), (0, 0))))]
    dq, dkn, dvn, dk, dv = (to_dev(b) for b in bits)
    lay = B.CacheLayout(Hq, Hkv, 128, 128, (n + 1) * 128, 0.05)
    out = torch.zeros(Hq, 128, device="cuda")
    B.check(B.lookm_decode_step(dq, dkn, dvn, dk, dv, n, lay, out, B.alloc_decode_workspace(lay)))
    f = [synth.bf16_to_f32(b) for b in bits]
    ref, _, _ = orc.decode_step(f[0], f[1], f[2], f[3][:, :n], f[4][:, :n], scale=0.05)
    got = out.cpu().numpy().astype(np.float64)
    assert np.all(got[:, 7] == np.inf) and np.all(got[:, 9] == -np.inf)
    rest = np.ones(128, dtype=bool)
    rest[[7, 9]] = False
    assert close(got[:, rest], ref[:, rest]).all()


@pytest.mark.parametrize("Hq,Hkv,n", [(1, 1, 17), (8, 8, 16), (12, 12, 409), (13, 13, 700), (32, 32, 18), (32, 32, 4095),
                                      (48, 48, 401), (64, 16, 100), (24, 3, 50), (40, 40, 520)])
def test_splits_added_up_by_a_cluster(B, Hq, Hkv, n):
    """Clusters of 2, 4 and 8 CTAs, scalar and grouped queries, with splits that get no row at all
    (17 rows over 8 splits of 3); one launch."""
    run_step(B, Hq, Hkv, n, n + 1, n % 2 == 0, seed=790 + n + Hq)
    assert B.lookm_last_launch_count() == (1 if n != 520 else 2)


@pytest.mark.parametrize("Hq,Hkv,n", [(32, 16, 3276), (64, 32, 409), (8, 4, 9000), (48, 8, 60), (64, 32, 5000), (16, 1, 700)])
def test_grouped_queries_one_or_two_heads_at_a_time(B, Hq, Hkv, n):
    """Groups whose heads are cheaper taken one by one or two by two: clusters and split records."""
    run_step(B, Hq, Hkv, n, n + 1, n % 2 == 0, seed=830 + n)


@pytest.mark.parametrize("group", [2, 3, 4, 5, 6, 7, 8, 12, 16])
def test_batches_of_grouped_queries_at_the_edges_of_sixteen_row_steps(B, group):
    """Enough requests for the tensor-core kernel whatever the rows: caches that end just before, at and after
    the sixteen rows of a warp's step and the sixty-four of a CTA's, the appended row in any of them."""
    import torch
    Hkv, f = 8, synth.bf16_to_f32
    lens = [0, 1, 7, 14, 15, 16, 17, 30, 31, 32, 47, 62, 63, 64, 65, 79, 80, 126, 127, 128, 129, 200, 255, 256, 257] * 3
    begins = np.concatenate([[0], np.cumsum([n + 1 for n in lens])]).tolist()
    ck_b, cv_b = _bits((begins[-1], Hkv, 128), (840, group)), _bits((begins[-1], Hkv, 128), (841, group))
    q_b, kn_b, vn_b = (_bits((len(lens), h, 128), (842 + i, group)) for i, h in enumerate((Hkv * group, Hkv, Hkv)))
    dk, dv, q, kn, vn = (to_dev(t) for t in (ck_b, cv_b, q_b, kn_b, vn_b))
    lay = B.CacheLayout(Hkv * group, Hkv, 128, Hkv * 128, 128, 0.2)
    out = torch.full((len(lens), Hkv * group, 128), np.nan, device="cuda")
    B.check(B.lookm_decode_step_varlen(q, kn, vn, dk, dv, begins[:-1], lens, lay, out, B.alloc_decode_workspace(lay, len(lens))))
    got = out.cpu().numpy().astype(np.float64)
    for r, n in enumerate(lens):
        a = begins[r]
        ref, _, _ = orc.decode_step(f(q_b[r]), f(kn_b[r]), f(vn_b[r]), f(ck_b[a:a + n]).transpose(1, 0, 2),
                                    f(cv_b[a:a + n]).transpose(1, 0, 2), scale=0.2)
        assert close(got[r], ref).all(), (r, n)
        assert torch.equal(dk[a + n], kn[r]) and torch.equal(dv[a + n], vn[r])


def records_of_shares(lens, q_heads, sms):
    """Partial results that the CTAs of a step in equal shares leave behind, by their place in the workspace: the
    steps of 64 rows of all (request, query head), in a row, are dealt to two CTAs per SM; a CTA whose share holds
    a unit in part writes the first of its two records if the share begins with the unit or inside it, else the second."""
    records = set()
    for chunk in range(0, len(lens), 96):                # requests that one launch carries
        units = [n // 64 + 1 for n in lens[chunk:chunk + 96] for _ in range(q_heads)]
        ends = np.cumsum(units)
        ctas = min(2 * sms, int(ends[-1]))
        shares = np.concatenate([[0], np.cumsum([int(ends[-1]) // ctas + (c < int(ends[-1]) % ctas) for c in range(ctas)])])
        for end, steps in zip(ends.tolist(), units):
            first, last = (int(np.searchsorted(shares, x, side="right")) - 1 for x in (end - steps, end - 1))
            if first < last:
                records |= {2 * c + int(c == first and shares[c] < end - steps) for c in range(first, last + 1)}
    return records


# (The planner goes by estimated times: where a refit of these sends a case another way, `shared` tells.)
@pytest.mark.parametrize("lens,heads,group,ranked,shared", [
    ([0, 1, 31, 40, 62, 63, 64, 65, 126, 127, 128, 129] * 9, 24, 1, False, True),      # more requests than one launch carries
    ([40] * 64, 32, 1, True, True),                      # units of one step: none is divided
    ([40] * 63 + [200], 32, 1, True, True),
    ([7000, 63, 64, 2000], 32, 1, False, True),          # units that many CTAs share beside units of a single step
    ([1600], 76, 1, True, True),                         # one request, a head per 3.9 CTAs
    ([4000], 76, 1, False, True),
    ([32768], 40, 1, True, True),                        # a head per 7.4 CTAs
    ([3166, 307], 5, 11, True, True),                    # grouped queries, one head at a time
    ([700, 3000, 64], 3, 13, False, True),
    ([13, 13, 32, 874], 6, 5, True, True),
    # whole splits, where a share of short units would last longest or two launches would take longer
    ([61, 1582, 4390, 3260, 2685, 2120, 3375, 841, 2736], 32, 1, True, False),
    ([968, 54, 847, 280, 513, 756, 184, 867, 453, 106, 997, 399, 1168, 641, 613, 119, 850], 8, 1, False, False),
    ([20031], 40, 1, True, False),
    ([628, 52, 10], 4, 11, False, False),
    ([8000], 32, 3, False, False),                       # tensor cores
    ([5000, 100, 5000], 20, 2, False, False)])
def test_equal_shares_of_all_rows(B, lens, heads, group, ranked, shared):
    """CTAs whose shares begin and end anywhere in a unit: units of less than a step to hundreds of steps, the
    appended row in the last step or in one of its own; `heads` KV heads, [heads, rows, 128] or packed."""
    import torch
    f, n_req, hq = synth.bf16_to_f32, len(lens), heads * group
    begins = np.concatenate([[0], np.cumsum([n + 1 for n in lens])]).tolist()
    shape = (heads, begins[-1], 128) if ranked else (begins[-1], heads, 128)
    gen = torch.Generator(device="cuda").manual_seed(len(lens) + heads)
    dk, dv, q, kn, vn = (torch.randn(*s_, 128, generator=gen, device="cuda").bfloat16()
                         for s_ in (shape[:2], shape[:2], (n_req, hq), (n_req, heads), (n_req, heads)))
    lay = B.CacheLayout(hq, heads, 128, *((128, begins[-1] * 128) if ranked else (heads * 128, 128)), 0.0)
    ws = B.alloc_decode_workspace(lay, n_req)
    outs = []
    by_head = lambda t: t if ranked else t.transpose(0, 1)
    before_k, before_v = dk.clone(), dv.clone()
    for last in (False, False, True):
        ws.fill_(255) if last else ws.random_(0, 255)    # nothing in the workspace counts
        out = torch.full((n_req, hq, 128), np.nan, device="cuda")
        B.check(B.lookm_decode_step_varlen(q, kn, vn, dk, dv, begins[:-1], lens, lay, out, ws))
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    words = ws.view(torch.int32)
    records = words[:words.numel() // 130 * 130].view(-1, 130)           # reference, sum and 128 features
    written = set((records != -1).any(1).nonzero()[:, 0].tolist())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (written == records_of_shares(lens, hq, sms)) == shared, "another kernel took the step"
    K, V = by_head(dk).double(), by_head(dv).double()
    untouched = torch.ones(begins[-1], dtype=torch.bool, device="cuda")
    for r, n in enumerate(lens):
        a = begins[r]
        assert torch.equal(by_head(dk)[:, a + n], kn[r]) and torch.equal(by_head(dv)[:, a + n], vn[r])
        untouched[a + n] = False
        s_ = torch.einsum("hgd,hnd->hgn", q[r].double().view(heads, group, 128), K[:, a:a + n + 1]) / 128 ** 0.5
        ref = torch.einsum("hgn,hnd->hgd", s_.softmax(-1), V[:, a:a + n + 1]).reshape(hq, 128)
        assert ((outs[0][r].double() - ref).abs() <= 1e-3 * ref.abs() + 1e-5).all(), (r, n)
    assert torch.equal(by_head(dk)[:, untouched], by_head(before_k)[:, untouched])
    assert torch.equal(by_head(dv)[:, untouched], by_head(before_v)[:, untouched])


def test_long_cache_is_cut_into_many_splits(B):
    # 2 KV heads x 20001 rows: about 150 splits per head, combined by the last CTA to arrive
    run_step(B, 8, 2, 20000, 20001, False, seed=701)
    run_step(B, 2, 2, 5000, 5002, True, seed=702, scale=0.3)


def test_peaked_softmax_and_custom_scale(B):
    # queries 6x larger: a few rows take nearly all the weight, references move along the cache
    run_step(B, 4, 2, 3000, 3001, False, seed=703, q_scale=6.0)
    run_step(B, 4, 2, 300, 301, True, seed=704, scale=1.0)


def test_batch_of_requests_with_their_own_lengths(B):
    import torch
    n_req, Hq, Hkv = 100, 4, 2                           # more requests than one launch carries
    lens = synth.uniform_int(synth.stream_key(710), n_req, 0, 400).astype(int).tolist()
    lens[3], lens[50] = 0, 2500
    caps = [n + 1 for n in lens]
    begins = np.concatenate([[0], np.cumsum(caps)])[:-1].tolist()
    rows = sum(caps)
    ck_b, cv_b = _bits((rows, Hkv, 128), (711,)), _bits((rows, Hkv, 128), (712,))
    q_b, kn_b, vn_b = _bits((n_req, Hq, 128), (713,)), _bits((n_req, Hkv, 128), (714,)), _bits((n_req, Hkv, 128), (715,))
    dk, dv, q, kn, vn = (to_dev(t) for t in (ck_b, cv_b, q_b, kn_b, vn_b))
    lay = B.CacheLayout(Hq, Hkv, 128, Hkv * 128, 128, 0.0)
    ws = B.alloc_decode_workspace(lay, n_req)
    out = torch.full((n_req, Hq, 128), np.nan, dtype=torch.float32, device="cuda")
    B.check(B.lookm_decode_step_varlen(q, kn, vn, dk, dv, begins, lens, lay, out, ws))
    torch.cuda.synchronize()
    # two launches of at most 96 requests, each followed by one combine launch if any of its
    # requests was cut into several splits
    assert 2 <= B.lookm_last_launch_count() <= 4
    got = out.cpu().numpy().astype(np.float64)
    f = synth.bf16_to_f32
    K, V = f(ck_b), f(cv_b)
    for r in range(n_req):
        a, n = begins[r], lens[r]
        ref, ck2, _ = orc.decode_step(f(q_b[r]), f(kn_b[r]), f(vn_b[r]), K[a:a + n].transpose(1, 0, 2),
                                      V[a:a + n].transpose(1, 0, 2))
        assert close(got[r], ref).all(), r
        assert torch.equal(dk[a + n], kn[r]) and torch.equal(dv[a + n], vn[r])
    untouched = np.ones(rows, dtype=bool)
    untouched[[b + n for b, n in zip(begins, lens)]] = False
    sel = torch.from_numpy(untouched).cuda()
    assert torch.equal(dk[sel], to_dev(ck_b)[sel]) and torch.equal(dv[sel], to_dev(cv_b)[sel])


def test_compress_then_generate_three_tokens(B):
    """The path's own output as the cache.  The oracle compresses the prompt itself and its rows,
    rounded to bf16, are the cache of the oracle's three generation steps.  The GPU runs the same
    steps twice: on a copy of exactly those rows (tight tolerance: same bits in, Eq. 2-3 alone),
    and chained after its own compression into a cache with room to grow (merged rows may differ
    from the oracle's by the 2e-2 of the merge tolerance, and so may the attention output)."""
    import torch
    L, Hq, Hkv, budget, window, steps = 1500, 8, 2, 300, 32, 3
    w = synth.tiny(L, Hq, Hkv, budget, window, 2, image_spans=[(100, 700), (800, 1400)], seed=41)
    qb, kb, vb = synth.layer_tensors(w)
    f = synth.bf16_to_f32
    res = orc.compress_layer(f(qb), f(kb), f(vb), w.requests[0].mask, budget, window, 2, threads=2,
                             score_dtype=np.float32)
    ok_bits = synth.f32_to_bf16_bits(np.stack(res["out_k"]).astype(np.float32))     # [Hkv, budget, 128]
    ov_bits = synth.f32_to_bf16_bits(np.stack(res["out_v"]).astype(np.float32))
    cap = budget + steps
    clay = B.CacheLayout(Hq, Hkv, 128, 128, cap * 128, 0.0)
    dws = B.alloc_decode_workspace(clay)
    # GPU cache 1: the oracle's rows.  GPU cache 2: the GPU's own compression.
    c1k = torch.zeros(Hkv, cap, 128, dtype=torch.bfloat16, device="cuda")
    c1v = torch.zeros_like(c1k)
    c1k[:, :budget], c1v[:, :budget] = to_dev(ok_bits), to_dev(ov_bits)
    q, k, v = to_dev(qb), to_dev(kb), to_dev(vb)
    lay = B.make_layout(q, k)
    ws = B.alloc_workspace(lay, [L])
    c2k, c2v = torch.zeros_like(c1k), torch.zeros_like(c1k)
    st, out_len = B.lookm_compress_layer_opt(q, k, v, torch.from_numpy(w.requests[0].mask).cuda(), L, budget,
                                             window, 2, lay, B.make_options(out_stride_head=cap * 128),
                                             c2k, c2v, ws)
    B.check(st)
    assert out_len == budget and B.lookm_device_status(ws) == B.OK
    ref_k, ref_v = f(ok_bits), f(ov_bits)
    out1 = torch.zeros(Hq, 128, dtype=torch.float32, device="cuda")
    out2 = torch.zeros_like(out1)
    for t in range(steps):
        q_b, kn_b, vn_b = _bits((Hq, 128), (720, t, 1)), _bits((Hkv, 128), (720, t, 2)), _bits((Hkv, 128), (720, t, 3))
        dq, dkn, dvn = to_dev(q_b), to_dev(kn_b), to_dev(vn_b)
        B.check(B.lookm_decode_step(dq, dkn, dvn, c1k, c1v, budget + t, clay, out1, dws))
        B.check(B.lookm_decode_step(dq, dkn, dvn, c2k, c2v, budget + t, clay, out2, dws))
        torch.cuda.synchronize()
        ref, ref_k, ref_v = orc.decode_step(f(q_b), f(kn_b), f(vn_b), ref_k, ref_v)
        assert close(out1.cpu().numpy().astype(np.float64), ref).all(), t
        assert np.abs(out2.cpu().numpy().astype(np.float64) - ref).max() <= 2e-2, t
    assert np.array_equal(c1k.float().cpu().numpy(), ref_k) and np.array_equal(c1v.float().cpu().numpy(), ref_v)
    assert torch.equal(c2k[:, budget:], c1k[:, budget:]) and torch.equal(c2v[:, budget:], c1v[:, budget:])


@pytest.mark.parametrize("ratio", [1.0, 0.2, 0.05])
def test_7b_shape_cache_at_the_papers_three_budgets(B, ratio):
    """32 heads over a cache of 100 %, 20 % and 5 % of the 8192-token prompt (the budgets of the
    paper's speed and memory table), every head against the oracle."""
    run_step(B, 32, 32, int(ratio * 8192), int(ratio * 8192) + 8, False, seed=730 + int(100 * ratio))
