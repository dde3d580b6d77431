"""The KV cache held as weights (paper Section 3.8) against the CPU oracle, through the C-ABI, on a B200: the
protocol of the paper's LLM benchmark, 1024 prefill tokens then 256 decode steps (Section 4.2), for one KV head of
a grouped-query model (4 query heads per KV head, d_h = 128)."""
import numpy as np
import pytest

from oracle import qlinear_oracle as O
from workloads import generators as gen

pytestmark = pytest.mark.gpu

CACHE, DH, GROUP = 1280, 128, 4


@pytest.fixture(scope="module")
def P(_built_library):
    import paper_2505_00232_b200 as P
    return P


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    return torch


def tensors(seed, T):
    k = gen.normal_fp16(seed, 1, (T, DH))
    v = gen.normal_fp16(seed, 2, (T, DH))
    v[5, :] = 0                                         # a zero vector: stored as zeros with scale 1
    k[7, :] *= np.float16(40.0)                         # per-token scales really differ
    return k, v


def test_append_writes_exactly_the_oracles_integers_and_scales(P, torch):
    k, v = tensors(811, CACHE)
    cache = P.KVCache(CACHE, DH)
    kd, vd = torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda()
    cache.append(kd[:1024], vd[:1024])                  # prefill: 1024 tokens in one call
    for t in range(1024, CACHE):                        # decode: one token per step
        cache.append(kd[t:t + 1], vd[t:t + 1])
    torch.cuda.synchronize()
    assert cache.length == CACHE and cache.k.device_status() == (0, 0)
    k_q, k_s = O.kv_quantize_rows(k)
    v_q, v_s = O.kv_quantize_rows(v)
    assert (cache.k.debug_unpack().cpu().numpy() == k_q).all()           # K cache: O = positions, I = d_h
    assert (cache.v.debug_unpack().cpu().numpy() == v_q.T).all()         # V cache: O = d_h, I = positions
    _, ks_blob = P.qlinear_unpack(cache.k.desc, cache.k.packed.cpu().numpy())
    assert (ks_blob.reshape(-1).view(np.uint16) == k_s.view(np.uint16)).all()
    assert (cache.v_scale.cpu().numpy().view(np.uint16) == v_s.view(np.uint16)).all()


@pytest.mark.parametrize("R,T", [(GROUP, 1280), (GROUP, 1031), (1, 200), (GROUP * 128, 1024)],
                         ids=["decode-full-cache", "decode-partial-cache", "one-row", "prefill-512-rows"])
def test_attention_products_match_the_oracle(P, torch, R, T):
    """scores = Q K^T and out = P V through the linear kernels (R = S * h_q / h_kv query rows of one KV head),
    inside the linear layer's tolerance; positions beyond the cache length score exactly 0."""
    k, v = tensors(900 + T, T)
    qry = gen.normal_fp16(900 + T, 3, (R, DH))
    cache = P.KVCache(CACHE, DH)
    cache.append(torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda())
    sc = cache.scores(torch.from_numpy(qry).cuda())
    torch.cuda.synchronize()
    sc_np = sc.cpu().numpy()
    assert (sc_np[:, T:] == 0).all()
    # probabilities: a softmax over the live positions (computed here in fp64: masking and softmax are the caller's)
    z = sc_np[:, :T].astype(np.float64) / np.sqrt(DH)
    p = np.exp(z - z.max(axis=1, keepdims=True))
    prob = np.zeros((R, CACHE), np.float16)
    prob[:, :T] = (p / p.sum(axis=1, keepdims=True)).astype(np.float16)
    out = cache.output(torch.from_numpy(prob).cuda())
    torch.cuda.synchronize()
    sc64, A_sc, out64, A_out = O.kv_attention(qry, k, v, prob[:, :T])
    ok, rel, worst = O.check_against(sc_np[:, :T], sc64, A_sc)
    assert ok, ("scores", rel, worst)
    ok, rel, worst = O.check_against(out.cpu().numpy(), out64, A_out)
    assert ok, ("output", rel, worst)


def test_append_argument_errors(P, torch):
    cache = P.KVCache(256, 64)
    a = torch.zeros((200, 64), dtype=torch.float16, device="cuda")
    cache.append(a, a)
    with pytest.raises(P.QLinearError):
        cache.append(a, a)                              # 400 > 256 positions
    other = P.KVCache(256, 32)
    import ctypes
    vp = ctypes.c_void_p
    assert P.lib.qlinear_kv_append(cache.k._h, other.v._h, vp(a.data_ptr()), vp(a.data_ptr()), vp(cache.v_scale.data_ptr()), 0, 1, None) == 1


@pytest.mark.parametrize("n_heads", [3, 8, 11])
def test_all_heads_in_one_launch_match_the_per_head_calls(P, torch, n_heads):
    """qlinear_kv_*_heads (every KV head of a layer in one launch, value scales folded inside the decode kernel) against
    the per-head calls: the same cache bytes and scales, the same score and output bits; and the output against the
    oracle.  11 heads: more than one launch's worth."""
    T, R = 1031, GROUP
    ks, vs, qs = [], [], []
    for h in range(n_heads):
        k, v = tensors(1200 + h, T)
        ks.append(k); vs.append(v); qs.append(gen.normal_fp16(1200 + h, 3, (R, DH)))
    k_all, v_all, q_all = (torch.from_numpy(np.stack(a)).cuda() for a in (ks, vs, qs))
    heads = P.KVHeads(n_heads, CACHE, DH)
    heads.append(k_all[:, :1024].contiguous(), v_all[:, :1024].contiguous())        # prefill
    for t in range(1024, T):                                                        # decode steps, strided input
        heads.append_raw(k_all[:, t].data_ptr(), v_all[:, t].data_ptr(), T * DH, DH, 1)
    singles = [P.KVCache(CACHE, DH) for _ in range(n_heads)]
    for h, c in enumerate(singles):
        c.append(k_all[h], v_all[h])
    torch.cuda.synchronize()
    assert heads.length == T
    for h in range(n_heads):
        assert torch.equal(heads.heads[h].k.packed, singles[h].k.packed)
        assert torch.equal(heads.heads[h].v.packed, singles[h].v.packed)
        assert torch.equal(heads.heads[h].v_scale, singles[h].v_scale)
    sc = heads.scores(q_all)
    z = sc[:, :, :T].double() / np.sqrt(DH)
    prob = torch.zeros((n_heads, R, CACHE), dtype=torch.float16, device="cuda")
    prob[:, :, :T] = torch.softmax(z, dim=2).half()
    out = heads.output(prob)
    torch.cuda.synchronize()
    assert heads.heads[0].k.device_status() == (0, 0)
    for h in range(n_heads):
        assert torch.equal(sc[h], singles[h].scores(q_all[h]))
        # the product with the scales as a pass of its own (one rounding to fp16), then the plain layer
        folded = (prob[h].float() * singles[h].v_scale.float()[None, :]).half()
        assert torch.equal(out[h], singles[h].v.forward(folded))
        assert torch.equal(out[h], singles[h].output(prob[h]))
        _, _, out64, A_out = O.kv_attention(qs[h], ks[h], vs[h], prob[h, :, :T].cpu().numpy())
        ok, rel, worst = O.check_against(out[h].cpu().numpy(), out64, A_out)
        assert ok, ("output", h, rel, worst)


def test_heads_argument_errors(P, torch):
    heads = P.KVHeads(2, 256, 64)
    big = torch.zeros((2, 9, 256), dtype=torch.float16, device="cuda")
    with pytest.raises(P.QLinearError):
        heads.output(big)                               # 9 query rows: not a decode-sized product
    with pytest.raises(P.QLinearError):
        heads.append(torch.zeros((3, 1, 64), dtype=torch.float16, device="cuda"), torch.zeros((3, 1, 64), dtype=torch.float16, device="cuda"))


@pytest.mark.parametrize("d_h,cache,n_heads,R", [(128, 10240, 8, 4), (64, 20000 // 32 * 32, 8, 1), (256, 9632, 8, 8), (128, 25632, 3, 5)],
                         ids=["dh128", "dh64-one-row", "dh256-eight-rows", "three-heads-ragged"])
def test_scores_over_a_long_cache_match_the_per_head_calls(P, torch, d_h, cache, n_heads, R):
    """More than one wave of row super-blocks: the score product of all heads runs on the persistent short-K kernel
    (a CTA walks over super-blocks, the next one's bytes in flight).  Same bits as the per-head calls of the ordinary
    decode kernel; cache lengths that are not a multiple of 128; positions beyond the filled part score 0."""
    T = cache - 777
    rng = np.random.default_rng(d_h + cache)
    k = (rng.standard_normal((n_heads, T, d_h)) * rng.uniform(0.2, 3.0, size=(n_heads, T, 1))).astype(np.float16)
    q = rng.standard_normal((n_heads, R, d_h)).astype(np.float16)
    kd, qd = torch.from_numpy(k).cuda(), torch.from_numpy(q).cuda()
    heads = P.KVHeads(n_heads, cache, d_h)
    heads.append(kd, kd)
    sc = heads.scores(qd)
    torch.cuda.synchronize()
    assert heads.heads[0].k.device_status() == (0, 0)
    assert (sc[:, :, T:] == 0).all()
    for h in range(n_heads):
        if d_h <= 128:                                  # (at d_h = 256 the per-head call splits K: another order of sums)
            assert torch.equal(sc[h], heads.heads[h].scores(qd[h]))
        k_q, k_s = O.kv_quantize_rows(k[h])
        y64, A, _ = O.linear(q[h], k_q, k_s.reshape(-1, 1), 0)
        ok, rel, worst = O.check_against(sc[h, :, :T].cpu().numpy(), y64, A)
        assert ok, (h, rel, worst)


def test_small_launches_are_planned_without_clusters(P, torch):
    """A cluster launch with its cluster-wide barriers costs about a microsecond: a forward call on a layer of a few MB is planned
    without one, large layers with a long K still take clusters.  (The value product over a cache has a plan of its own,
    test_value_product_is_planned_for_one_wave.)"""
    import ctypes

    def plan(lin, M):
        out = (ctypes.c_int32 * 8)()
        assert P.lib.qlinear_debug_plan(lin._h, M, out, 8) == 8
        return {"grid": out[1], "cl": out[2], "ks_cta": out[3], "cps": out[4]}
    v = P.KVCache(CACHE, DH).v                           # N = 128, K = 1280: 164 KB
    assert plan(v, 4)["cl"] == 1
    big = P.QLinear(P.Desc(4096, 14336, 8, 0), torch.zeros(P.qlinear_packed_size(P.Desc(4096, 14336, 8, 0)), dtype=torch.uint8, device="cuda"))
    assert plan(big, 1)["cl"] > 1


@pytest.mark.parametrize("R", [GROUP, 64, 256])
def test_products_see_the_tokens_appended_just_before(P, torch, R):
    """append, scores, output enqueued back to back (a captured graph, replayed on new tokens), against the same calls with the
    host waiting in between: the products request cache bytes ahead of their stream dependency, so the append may not let
    them start before its bytes are written."""
    n_heads, T = 8, 1000
    k0, v0 = tensors(1700, T)
    start = torch.from_numpy(np.stack([k0] * n_heads)).cuda(), torch.from_numpy(np.stack([v0] * n_heads)).cuda()
    pair = [P.KVHeads(n_heads, CACHE, DH) for _ in range(2)]
    for kv in pair:
        kv.append(*start)
    q = torch.randn((n_heads, R, DH), device="cuda").half()
    prob = torch.full((n_heads, R, CACHE), 2.0 ** -10, dtype=torch.float16, device="cuda")
    kn, vn = (torch.zeros((n_heads, 5, DH), dtype=torch.float16, device="cuda") for _ in range(2))

    def step(kv, wait):
        kv.length = T
        kv.append(kn, vn)
        wait()
        sc = kv.scores(q)
        wait()
        return sc, [c.output(prob[i]) for i, c in enumerate(kv.heads)]
    step(pair[0], lambda: None)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sc, out = step(pair[0], lambda: None)
    for _ in range(20):
        kn.copy_(torch.randn_like(kn) * 3)
        vn.copy_(torch.randn_like(vn) * 3)
        graph.replay()
        torch.cuda.synchronize()
        sc_w, out_w = step(pair[1], torch.cuda.synchronize)
        torch.cuda.synchronize()
        assert torch.equal(sc, sc_w) and all(torch.equal(a, b) for a, b in zip(out, out_w))


@pytest.mark.parametrize("n_heads,d_h,cache,R", [(1, 64, 32, 1), (1, 64, 992, 8), (3, 128, 2048, 5), (8, 128, 4128, 4), (2, 256, 8192, 7)])
def test_value_product_over_slices_of_any_length(P, torch, n_heads, d_h, cache, R):
    """The decode kernel of the value product: fewer chunks than warps, a ring that is not a multiple of the slice, slices that
    end early, with and without a split over a cluster."""
    rng = np.random.default_rng(cache + R)
    v = (rng.standard_normal((n_heads, cache, d_h)) * rng.uniform(0.2, 3.0, size=(n_heads, cache, 1))).astype(np.float16)
    prob = (rng.random((n_heads, R, cache)) / cache).astype(np.float16)
    heads = P.KVHeads(n_heads, cache, d_h)
    vd = torch.from_numpy(v).cuda()
    heads.append(vd, vd)
    out = heads.output(torch.from_numpy(prob).cuda())
    torch.cuda.synchronize()
    assert heads.heads[0].v.device_status() == (0, 0)
    for h in range(n_heads):
        v_q, v_s = O.kv_quantize_rows(v[h])
        folded = (prob[h].astype(np.float32) * v_s.astype(np.float32)).astype(np.float16)
        y64, A, _ = O.kv_output(folded, np.ascontiguousarray(v_q.T), np.ones(d_h, np.float16))
        ok, rel, worst = O.check_against(out[h].cpu().numpy(), y64, A)
        assert ok, (h, rel, worst)


@pytest.mark.parametrize("n_heads,d_h,cache,T,R", [(3, 64, 96, 90, 9), (1, 256, 992, 992, 17), (8, 128, 1280, 1031, 33), (11, 128, 160, 130, 100), (2, 64, 8192, 8000, 65), (2, 128, 4096, 3256, 1024)])
def test_scores_of_many_rows(P, torch, n_heads, d_h, cache, T, R):
    """The kernel of the score product for more than 8 query rows: token blocks of 16, 32 and 64 with a remainder, a last
    super-block that is not full, CTAs whose range of tiles spans heads; per head and all heads in one launch agree."""
    rng = np.random.default_rng(cache + R)
    k = (rng.standard_normal((n_heads, T, d_h)) * rng.uniform(0.2, 3.0, size=(n_heads, T, 1))).astype(np.float16)
    q = rng.standard_normal((n_heads, R, d_h)).astype(np.float16)
    heads = P.KVHeads(n_heads, cache, d_h)
    kd, qd = torch.from_numpy(k).cuda(), torch.from_numpy(q).cuda()
    heads.append(kd, kd)
    sc = heads.scores(qd)
    torch.cuda.synchronize()
    assert heads.heads[0].k.device_status() == (0, 0)
    assert (sc[:, :, T:] == 0).all()
    for h in range(n_heads):
        assert torch.equal(sc[h], heads.heads[h].scores(qd[h]))
        k_q, k_s = O.kv_quantize_rows(k[h])
        y64, A, _ = O.linear(q[h], k_q, k_s.reshape(-1, 1), 0)
        ok, rel, worst = O.check_against(sc[h, :, :T].cpu().numpy(), y64, A)
        assert ok, (h, rel, worst)


@pytest.mark.parametrize("d_h,cache,R", [(64, 96, 1), (128, 1280, 4), (256, 992, 8), (256, 9632, 5)])
def test_scores_of_one_head_are_those_of_all_heads(P, torch, d_h, cache, R):
    """One head's scores come from the kernel that serves all heads, K undivided: the same bits at every head dimension."""
    rng = np.random.default_rng(d_h + cache + R)
    k = rng.standard_normal((2, cache, d_h)).astype(np.float16)
    q = rng.standard_normal((2, R, d_h)).astype(np.float16)
    heads = P.KVHeads(2, cache, d_h)
    kd, qd = torch.from_numpy(k).cuda(), torch.from_numpy(q).cuda()
    heads.append(kd, kd)
    sc = heads.scores(qd)
    for h in range(2):
        assert torch.equal(sc[h], heads.heads[h].scores(qd[h]))
        k_q, k_s = O.kv_quantize_rows(k[h])
        y64, A, _ = O.linear(q[h], k_q, k_s.reshape(-1, 1), 0)
        ok, rel, worst = O.check_against(sc[h].cpu().numpy(), y64, A)
        assert ok, (h, rel, worst)
    assert heads.heads[0].k.device_status() == (0, 0)


@pytest.mark.parametrize("n_heads,d_h,cache", [(1, 64, 32), (8, 128, CACHE), (1, 128, 2048), (1, 128, 8192), (2, 128, 32768), (1, 256, 32768), (3, 128, 32768), (8, 128, 32768), (8, 256, 16384), (11, 64, 16384)])
def test_value_product_is_planned_for_one_wave(P, torch, n_heads, d_h, cache):
    """The launch that the value product makes: no clusters for a cache of up to 2048 positions, a split beyond where the row-blocks
    leave SMs idle, and never more clusters than run at once (a second wave of them costs more than the split gains)."""
    import ctypes
    desc = P.Desc(d_h, cache, 8, 0)
    v = P.QLinear(desc, torch.zeros(P.qlinear_packed_size(desc), dtype=torch.uint8, device="cuda"))
    out = (ctypes.c_int32 * 4)()
    assert P.lib.qlinear_debug_plan_kv_output(v._h, n_heads, out, 4) == 4
    cl, cps, clusters, at_once = out
    assert clusters == min(n_heads, 8) * d_h // 16
    assert cl == 1 or clusters <= at_once
    assert cps * 16 * cl >= cache // 32 and (cl == 1 or cps >= 2)        # (16 warps per CTA)
    if cache <= 2048 or clusters * 2 > torch.cuda.get_device_properties(0).multi_processor_count:
        assert cl == 1
    elif cache >= 8192 and clusters <= 16:
        assert cl >= 4


@pytest.mark.parametrize("d_h,R", [(96, 200), (512, 100), (512, 200), (384, 300)])
def test_prefill_kernels_see_the_tokens_appended_just_before(P, torch, d_h, R):
    """Scores of many rows at the head dimensions that the prefill kernels serve (single CTA, CTA pair split along K): append and
    scores back to back, on tokens that change every time, against the same calls with the host waiting in between."""
    T, n_new = 700, 5
    caches = [P.KVCache(768, d_h) for _ in range(2)]
    start = torch.randn((T, d_h), device="cuda").half()
    for c in caches:
        c.append(start, start)
    q = torch.randn((R, d_h), device="cuda").half()
    for _ in range(30):
        kn = (torch.randn((n_new, d_h), device="cuda") * 3).half()
        torch.cuda.synchronize()
        got = []
        for c, wait in zip(caches, (lambda: None, torch.cuda.synchronize)):
            for factor in (0.5, 2.0, 1.0):
                c.length = T
                c.append(kn * factor, kn)
                wait()
                sc = c.scores(q)
            torch.cuda.synchronize()
            got.append(sc)
        assert torch.equal(*got)
    assert caches[0].k.device_status() == (0, 0)
    k_q, k_s = O.kv_quantize_rows(kn.cpu().numpy())
    y64, A, _ = O.linear(q.cpu().numpy(), k_q, k_s.reshape(-1, 1), 0)
    ok, rel, worst = O.check_against(got[0][:, T:T + n_new].cpu().numpy(), y64, A)
    assert ok, (rel, worst)


@pytest.mark.parametrize("n_heads,cache", [(8, 2048), (11, 1280), (8, 8192), (11, 4096)])
def test_value_product_of_all_heads_and_of_one(P, torch, n_heads, cache):
    """Up to 2048 positions K is undivided whatever the number of heads: the same bits.  Beyond, the split follows the number of
    heads in the launch: the same value up to the order of the fp32 sums, which two fp16 roundings of it bound."""
    rng = np.random.default_rng(n_heads + cache)
    v = torch.from_numpy(rng.standard_normal((n_heads, cache, DH)).astype(np.float16)).cuda()
    prob = (torch.rand((n_heads, 4, cache), device="cuda") / cache).half()
    heads = P.KVHeads(n_heads, cache, DH)
    heads.append(v, v)
    out = heads.output(prob)
    for h in range(n_heads):
        one = heads.heads[h].output(prob[h])
        if cache <= 2048:
            assert torch.equal(out[h], one)
        else:
            # |sum| <= A, the sum of the magnitudes: each order errs by at most (positions / 32 + 48) 2^-24 A before its rounding
            A = (prob[h].float() * heads.heads[h].v_scale.float()) @ (heads.heads[h].v.debug_unpack().float().abs().T)
            bound = 2.0 ** -10 * one.float().abs() + 2 * (cache / 32 + 48) * 2.0 ** -24 * A + 2.0 ** -24
            assert bool(((out[h].float() - one.float()).abs() <= bound).all())
