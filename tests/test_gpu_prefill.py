"""GPU causal prefill (mlkv_prefill, tcgen05 kernel) against the fp64 oracle's prefill.

Every layer of a model is prefilled in order (owner layers store the prompt's K/V, every layer
attends causally over its owner's slot); all rows of every prompt are compared.  Prompt lengths
straddle the 128-position blocks of the kernel; rows past a prompt's length must stay untouched.
A decode step then continues every sequence from the prefilled cache.
"""
import numpy as np
import pytest

import oracle
from mlkv_synth import gen
from tests.mlkv_cases import MAX_ABS, MEAN_ABS, errors, from_dev, to_dev

pytestmark = pytest.mark.gpu

EDGE_PROMPTS = [1, 127, 128, 129, 300]


def _prefill_model(owner, h, g, d, b, prompt_lens, s_max, max_seq, seed, cache, ref, nthreads=4):
    """Prefills every layer of the model on the GPU and in the oracle; returns the worst error."""
    import torch

    l = len(owner)
    prompt_lens = np.asarray(prompt_lens, dtype=np.int32)
    worst = (0.0, 0.0)
    for n in range(l):
        qb = gen.gen_bf16(seed, gen.TID_Q + n, range(b * s_max), h * d).reshape(b, s_max, h, d)
        kd = vd = None
        if owner[n] == n:
            kb = gen.gen_kv(seed, n, 0, b, g, s_max, d)
            vb = gen.gen_kv(seed, n, 1, b, g, s_max, d)
            kd, vd = to_dev(kb), to_dev(vb)
            ref.load_prefix(n, gen.bf16_bits_to_f64(kb), gen.bf16_bits_to_f64(vb), s_max)
        out = torch.full((b, s_max, h, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        cache.prefill(n, to_dev(qb), kd, vd, out, prompt_lens)
        torch.cuda.synchronize()
        expect = ref.prefill(n, gen.bf16_bits_to_f64(qb), prompt_lens, nthreads=nthreads)
        got = from_dev(out)
        for beta in range(b):
            S = int(prompt_lens[beta])
            assert np.isfinite(got[beta, :S]).all(), f"layer {n} seq {beta}: non-finite output"
            assert np.isnan(got[beta, S:]).all(), f"layer {n} seq {beta}: rows past the prompt written"
            mx, mean = errors(got[beta, :S], expect[beta, :S])
            assert mx <= MAX_ABS and mean <= MEAN_ABS, (n, beta, mx, mean)
            worst = (max(worst[0], mx), max(worst[1], mean))
    cache.sync_status()
    return worst


@pytest.mark.parametrize("name,owner,h,g", [
    ("mha", [0, 1, 2], 4, 4),
    ("gqa", [0, 1, 2], 12, 4),
    ("mqa", [0, 1], 12, 1),
    ("mlkv-block", [0, 0, 2, 2], 12, 3),
    ("mlkv-1", [0, 0, 0], 16, 1),
    ("non-uniform", [0, 0, 0, 3, 4, 4], 8, 2),
])
@pytest.mark.parametrize("d", [64, 128])
def test_prefill_maps_and_edges(name, owner, h, g, d):
    import paper_2406_09297_gb300 as mlkv
    b, s_max = len(EDGE_PROMPTS), 300
    with mlkv.MLKVCache(len(owner), h, d, owner, g, b, s_max) as cache:
        ref = oracle.OracleCache(owner, h, g, d, b, s_max)
        _prefill_model(owner, h, g, d, b, EDGE_PROMPTS, s_max, s_max, 51, cache, ref)


@pytest.mark.parametrize("d", [64, 128])
def test_prefill_long_prompts(d):
    # 16 blocks of 128 positions per prompt: the causal triangle's tiles, longest blocks first
    import paper_2406_09297_gb300 as mlkv
    owner, h, g, b, s_max = [0, 0], 12, 1, 2, 2048
    with mlkv.MLKVCache(2, h, d, owner, g, b, s_max) as cache:
        ref = oracle.OracleCache(owner, h, g, d, b, s_max)
        _prefill_model(owner, h, g, d, b, [2048, 1500], s_max, s_max, 52, cache, ref, nthreads=2)


@pytest.mark.parametrize("h,g,d,b,s_max", [
    (12, 1, 64, 23, 385),     # 1,104 units and fewer: several per persistent CTA, uneven rounds
    (12, 4, 128, 37, 300),    # groups of 3: blocks in pairs, units with and without a tile A
    (16, 4, 128, 40, 200),    # head pairs
    (5, 5, 64, 61, 129),      # 305 heads of prompts: one CTA takes a second unit
])
def test_prefill_units_beyond_one_wave(h, g, d, b, s_max):
    # More units than resident CTAs (152 SMs, two per SM at head_dim 64): every CTA runs several
    # units on one set of barriers, query buffers and tensor-memory columns.
    import paper_2406_09297_gb300 as mlkv
    lens = [s_max if i % 3 == 0 else 1 + (i * 97) % s_max for i in range(b)]
    with mlkv.MLKVCache(1, h, d, [0], g, b, s_max) as cache:
        ref = oracle.OracleCache([0], h, g, d, b, s_max)
        _prefill_model([0], h, g, d, b, lens, s_max, s_max, 55, cache, ref, nthreads=8)


def test_prefill_long_prompt_every_row():
    # A 6000-position prompt: 47 key tiles per query block, units of very different lengths.
    import paper_2406_09297_gb300 as mlkv
    owner, h, g, d = [0], 4, 1, 64
    with mlkv.MLKVCache(1, h, d, owner, g, 1, 6000) as cache:
        ref = oracle.OracleCache(owner, h, g, d, 1, 6000)
        _prefill_model(owner, h, g, d, 1, [6000], 6000, 6000, 54, cache, ref, nthreads=8)


def test_prefill_then_decode_continues():
    # The cache a prefill leaves is the cache decoding continues from (Sec. 4.5: a prompt, then
    # tokens one by one): one decode step at length prompt + 1 in every layer.
    import torch

    import paper_2406_09297_gb300 as mlkv
    owner, h, g, d, b = [0, 0, 2, 2], 12, 3, 64, 3
    prompts = np.array([100, 257, 40], dtype=np.int32)
    s_max, max_seq = 257, 320
    seed = 53
    with mlkv.MLKVCache(len(owner), h, d, owner, g, b, max_seq) as cache:
        ref = oracle.OracleCache(owner, h, g, d, b, max_seq)
        _prefill_model(owner, h, g, d, b, prompts, s_max, max_seq, seed, cache, ref)
        lens = prompts + 1
        owners = sorted(set(owner))
        qb = np.stack([gen.gen_q(seed + 7, n, b, h, d) for n in range(len(owner))])
        kn = np.stack([gen.gen_bf16(seed + 8, gen.TID_K + n, range(b * g), d).reshape(b, g, d)
                       for n in owners])
        vn = np.stack([gen.gen_bf16(seed + 8, gen.TID_V + n, range(b * g), d).reshape(b, g, d)
                       for n in owners])
        out = torch.full((len(owner), b, h, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        cache.decode_step(to_dev(qb), to_dev(kn), to_dev(vn), out, lens)
        torch.cuda.synchronize()
        for n in range(len(owner)):
            if owner[n] == n:
                k = owners.index(n)
                ref.append(n, gen.bf16_bits_to_f64(kn[k]), gen.bf16_bits_to_f64(vn[k]), lens)
            expect = ref.decode(n, gen.bf16_bits_to_f64(qb[n]), lens)
            mx, mean = errors(from_dev(out[n]), expect)
            assert mx <= MAX_ABS and mean <= MEAN_ABS, (n, mx, mean)
        cache.sync_status()


def test_prefill_rejects_bad_arguments():
    import torch

    import paper_2406_09297_gb300 as mlkv
    with mlkv.MLKVCache(2, 4, 64, [0, 0], 2, 2, 256) as cache:
        q = torch.zeros((2, 256, 4, 64), dtype=torch.bfloat16, device="cuda")
        kv = torch.zeros((2, 2, 256, 64), dtype=torch.bfloat16, device="cuda")
        out = torch.zeros_like(q)
        for lens in ([0, 5], [257, 5]):
            with pytest.raises(mlkv.MLKVError) as e:
                cache.prefill(0, q, kv, kv, out, lens)
            assert e.value.code == mlkv.MLKV_ERR_RANGE
        with pytest.raises(mlkv.MLKVError) as e:
            cache.prefill(0, q, None, None, out, [5, 5])   # an owner layer needs its K/V
        assert e.value.code == mlkv.MLKV_ERR_INVALID_ARG
        with pytest.raises(mlkv.MLKVError) as e:
            cache.prefill(1, q, None, None, q, [5, 5])     # out overlapping Q
        assert e.value.code == mlkv.MLKV_ERR_INVALID_ARG
        cache.prefill(1, q, None, None, out, [5, 5])       # a non-owner layer needs no K/V
        cache.sync_status()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("shared", ["K", "V"])
def test_prefill_out_over_prompt_kv(d, shared):
    # The outputs may be written over the prompt's own keys or values: an owner layer then stores
    # them before it attends.  Outputs and cache equal those with separate buffers, bit for bit.
    import torch

    import paper_2406_09297_gb300 as mlkv
    from tests.test_gpu_cache import _read_cache
    h = g = 4
    b, s_max, max_seq = 3, 700, 704
    prompts = np.array([700, 1, 333], dtype=np.int32)
    Q = to_dev(gen.gen_q(61, 0, b * s_max, h, d).reshape(b, s_max, h, d))
    kv = [to_dev(gen.gen_kv(61, 0, i, b, g, s_max, d)) for i in range(2)]
    results = []
    for overlap in (False, True):
        with mlkv.MLKVCache(1, h, d, [0], g, b, max_seq) as cache:
            K, V = (t.clone() for t in kv)
            out = torch.zeros((b, s_max, h, d), dtype=torch.bfloat16, device="cuda")
            if overlap:
                out = (K if shared == "K" else V).view(b, s_max, h, d)
            cache.prefill(0, Q, K, V, out, prompts)
            torch.cuda.synchronize()
            cache.sync_status()
            results.append(([out[i, :n].clone() for i, n in enumerate(prompts)],
                            _read_cache(cache, b, g, max_seq, d)[:, :, :, :, :s_max]))
    for x, y in zip(results[0][0], results[1][0]):
        assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert (results[0][1] == results[1][1]).all()


@pytest.mark.parametrize("d,h,b", [(64, 12, 520), (128, 24, 520)])
def test_prefill_more_units_than_one_launch(d, h, b):
    # More than 6,144 units: an owner layer's several launches over the prompt's K/V in place, then
    # the store behind the last, and the reader's launches over the slot.
    import paper_2406_09297_gb300 as mlkv
    s_max = 130
    lens = [1 + (i * 61) % s_max for i in range(b)]
    with mlkv.MLKVCache(2, h, d, [0, 0], 1 if d == 64 else 2, b, s_max) as cache:
        ref = oracle.OracleCache([0, 0], h, 1 if d == 64 else 2, d, b, s_max)
        _prefill_model([0, 0], h, 1 if d == 64 else 2, d, b, lens, s_max, s_max, 62, cache, ref,
                       nthreads=8)


@pytest.mark.parametrize("d,h,g", [(64, 12, 3), (128, 16, 4)])
def test_prefill_among_other_calls_without_a_wait(d, h, g):
    # A decode of the slot's old contents, the owner's prefill (K/V read in place, stored in its
    # tail), its reader's prefill over the slot, the owner's and the reader's decode and a whole step,
    # queued without a host wait: every output and the cache bit for bit as with one after each call.
    import torch

    import paper_2406_09297_gb300 as mlkv
    from tests.test_gpu_cache import _read_cache
    b, S, max_seq = 6, 900, 1000
    prompts = np.array([900, 1, 333, 128, 650, 257], dtype=np.int32)

    def rand(seed, *shape):
        gen_ = torch.Generator(device="cuda").manual_seed(seed)
        return torch.randn(shape, device="cuda", generator=gen_).bfloat16()

    with mlkv.MLKVCache(2, h, d, [0, 0], g, b, max_seq) as cache:
        q, pq = rand(1, 2, b, h, d), rand(2, 2, b, S, h, d)
        kn, vn = rand(3, 1, b, g, d), rand(4, 1, b, g, d)
        prompt_kv = [[rand(10 * r + i, b, g, S, d) for i in range(2)] for r in range(3)]
        outs = [torch.empty_like(q[0]) for _ in range(4)] + [torch.empty_like(q)]
        pouts = [torch.zeros_like(pq[0]) for _ in range(2)]

        def run(r, wait):
            def done():
                if wait:
                    torch.cuda.synchronize()
            K, V = prompt_kv[r]
            calls = [lambda: cache.decode_attention(1, q[1], outs[0], prompts),
                     lambda: cache.prefill(0, pq[0], K, V, pouts[0], prompts),
                     lambda: cache.prefill(1, pq[1], None, None, pouts[1], prompts),
                     lambda: cache.decode_attention(0, q[0], outs[1], prompts),
                     lambda: cache.append_decode_attention(0, kn[0], vn[0], q[0], outs[2], prompts + 1),
                     lambda: cache.decode_attention(1, q[1], outs[3], prompts + 1),
                     lambda: cache.decode_step(q, vn, kn, outs[4], prompts + 2)]
            for call in calls:
                call()
                done()
            torch.cuda.synchronize()
            return [x.clone() for x in outs + pouts] + [
                torch.from_numpy(_read_cache(cache, b, g, max_seq, d))]

        run(2, True)
        expect = [run(r, True) for r in range(3)]
        for rep in range(12):
            for x, y in zip(run(rep % 3, False), expect[rep % 3]):
                assert torch.equal(x.view(torch.int16), y.view(torch.int16)), rep
        cache.sync_status()


@pytest.mark.parametrize("what", ["KV", "own KV", "Q"])
def test_prefill_inputs_in_the_cache(what):
    # K and V in another slot, in the layer's own slot, and queries in another slot: the prompt is
    # stored before the attention.  Bits as from separate tensors.
    import torch

    import paper_2406_09297_gb300 as mlkv
    from tests.test_gpu_cache import _DevArray, _read_cache
    h, g, d, b, s = 8, 4, 64, 3, 300
    prompts = np.array([300, 1, 129], dtype=np.int32)
    Q = to_dev(gen.gen_q(63, 0, b * s, h, d).reshape(b, s, h, d))
    K, V = (to_dev(gen.gen_kv(63, 0, i, b, g, s, d)) for i in range(2))
    results = []
    for inside in (False, True):
        with mlkv.MLKVCache(2, h, d, [0, 1], g, b, s) as cache:
            cache.load_prefix(0, K, V, s)
            cache.load_prefix(1, K, V, s)
            n = b * g * s * d
            q, k, v = Q, K, V
            if inside and what != "Q":
                k, v = (torch.as_tensor(_DevArray(x, n), device="cuda").view(torch.bfloat16)
                        for x in cache.kv_ptr(0 if what == "own KV" else 1)[:2])
            elif what == "Q":
                q = torch.as_tensor(_DevArray(cache.kv_ptr(1)[0], 2 * n), device="cuda").view(
                    torch.bfloat16)[:Q.numel()].view(Q.shape)
                q.copy_(Q)
                if not inside:
                    q = Q
            out = torch.zeros((b, s, h, d), dtype=torch.bfloat16, device="cuda")
            cache.prefill(0, q, k, v, out, prompts)
            torch.cuda.synchronize()
            cache.sync_status()
            results.append((out, _read_cache(cache, b, g, s, d)))
    assert torch.equal(results[0][0].view(torch.int16), results[1][0].view(torch.int16))
    np.testing.assert_array_equal(results[0][1], results[1][1])
