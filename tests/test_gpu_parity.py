"""GPU decode attention against the fp64 oracle on small, fully checked cases.

Sizes span several tiles with ragged tails; the grid option forces segments to be split across
CTAs so that the partial-merge path runs; maps cover MHA, GQA, MQA, MLKV blocks and non-uniform
owner maps; head_dim 64 and 128; every tile variant.
"""
import numpy as np
import pytest

from tests.mlkv_cases import run_small_case

pytestmark = pytest.mark.gpu

TILE_EDGE_LENS = [1, 2, 15, 16, 17, 63, 64, 65, 127, 128, 129, 191, 256, 257, 300]


@pytest.mark.parametrize("d,tile", [(64, 128), (64, 64), (64, 256), (128, 64), (128, 128)])
@pytest.mark.parametrize("fused", [False, True])
def test_tile_edges_single_layer(d, tile, fused):
    b = len(TILE_EDGE_LENS)
    run_small_case([0], 4, 2, d, b, TILE_EDGE_LENS, 300, seed=11, options={"tile_tokens": tile},
                   fused=fused)


# The tcgen05 kernel (option "tc"): 128- and 256-position tiles, both head sizes, ragged lengths,
# split segments (stream-K records, inline and deferred merges) and DSMEM clusters.
@pytest.mark.parametrize("d,tile", [(64, 128), (64, 256), (128, 128)])
@pytest.mark.parametrize("fused", [False, True])
def test_tc_tile_edges(d, tile, fused):
    b = len(TILE_EDGE_LENS)
    run_small_case([0], 4, 2, d, b, TILE_EDGE_LENS, 300, seed=21,
                   options={"tile_tokens": tile, "tc": 1}, fused=fused, expect={"last_tc": 1})


@pytest.mark.parametrize("grid", [3, 7, 64, 600])
def test_tc_split_merges(grid):
    lens = [700, 1, 129, 1000]
    run_small_case([0, 0], 16, 1, 64, len(lens), lens, 1024, seed=22,
                   options={"grid": grid, "tile_tokens": 128, "tc": 1}, fused=True,
                   expect={"last_tc": 1})


@pytest.mark.parametrize("name,owner,h,g,d", [
    ("mha", [0, 1, 2], 4, 4, 64), ("gqa-mlkv", [0, 0, 0, 3, 3, 3], 12, 4, 64),
    ("mqa-g16", [0, 1], 16, 1, 128), ("non-uniform", [0, 0, 0, 3, 4, 4], 8, 2, 128)])
def test_tc_maps(name, owner, h, g, d):
    lens = [5, 130, 77, 260]
    run_small_case(owner, h, g, d, len(lens), lens, 320, seed=23,
                   options={"tc": 1, "tile_tokens": 128}, expect={"last_tc": 1})


def test_tc_cluster_merge():
    run_small_case([0, 0, 2], 12, 1, 64, 64, [2048] * 64, 2048, seed=24, fused=True,
                   options={"tc": 1}, expect={"last_tc": 1, "last_cluster_k": 2})


@pytest.mark.parametrize("lens", [[2048] * 4, [512, 1, 77, 2048], [600] * 3])
def test_default_tile_choice(lens):
    # the default tile length depends on the mean length; both choices are checked
    run_small_case([0, 0, 2], 12, 1, 64, len(lens), lens, 2048, seed=14, fused=True)


@pytest.mark.parametrize("grid", [1, 2, 3, 7, 64, 200, 600])
@pytest.mark.parametrize("fused", [False, True])
def test_split_merge_paths(grid, fused):
    # Many CTAs over few tiles: segments split across up to hundreds of CTAs (the largest grids
    # exceed the shared-memory merge capacity and take the fallback merge).
    lens = [700, 1, 129, 1000]
    run_small_case([0, 0], 16, 1, 64, len(lens), lens, 1024, seed=12,
                   options={"grid": grid, "tile_tokens": 64}, fused=fused)


@pytest.mark.parametrize("name,owner,h,g", [
    ("mha", [0, 1, 2], 4, 4),
    ("gqa", [0, 1, 2], 12, 4),
    ("mqa-g12", [0, 1], 12, 1),
    ("mqa-g16", [0, 1], 16, 1),
    ("mlkv-pairs", [0, 0, 2, 2], 12, 1),
    ("mlkv-1", [0, 0, 0, 0], 12, 1),
    ("gqa-mlkv", [0, 0, 0, 3, 3, 3], 12, 4),
    ("non-uniform", [0, 0, 0, 3, 4, 4], 8, 2),
    ("g8", [0, 0], 16, 2),
])
@pytest.mark.parametrize("d", [64, 128])
def test_maps(name, owner, h, g, d):
    lens = [5, 130, 77, 260]
    run_small_case(owner, h, g, d, len(lens), lens, 320, seed=13)


def test_random_fuzz():
    rng = np.random.default_rng(2024)
    for trial in range(12):
        l = int(rng.integers(1, 7))
        owner = []
        for n in range(l):
            o = int(rng.integers(0, n + 1))
            owner.append(o if (o == n or owner[o] == o) else n)
        h = int(rng.choice([1, 2, 3, 4, 6, 8, 12, 16]))
        divs = [x for x in range(1, h + 1) if h % x == 0]
        g = int(rng.choice(divs))
        d = int(rng.choice([64, 128]))
        b = int(rng.integers(1, 6))
        max_seq = int(rng.choice([1, 7, 64, 129, 333]))
        lens = rng.integers(1, max_seq + 1, size=b)
        opts = {"grid": int(rng.choice([0, 1, 5, 50]))}
        run_small_case(owner, h, g, d, b, lens, max_seq, seed=100 + trial, options=opts,
                       fused=bool(trial % 2))


def test_config1_full():
    from mlkv_synth import workloads
    w = workloads.config(1)
    run_small_case(w.owner, w.h, w.g, w.d, w.b, w.seq_lens(), w.max_seq, seed=w.seed)


def test_non_finite_cache_contents_beyond_length_do_not_leak():
    """Positions >= L of the cache may hold anything (here NaN); outputs stay finite."""
    import torch

    import paper_2406_09297_gb300 as mlkv
    from tests.mlkv_cases import errors, from_dev, to_dev
    import oracle
    from mlkv_synth import gen

    b, g, h, d, max_seq = 2, 1, 4, 64, 200
    lens = np.array([70, 3], dtype=np.int32)
    with mlkv.MLKVCache(1, h, d, [0], g, b, max_seq) as cache:
        kb = gen.gen_kv(5, 0, 0, b, g, max_seq, d)
        vb = gen.gen_kv(5, 0, 1, b, g, max_seq, d)
        kd, vd = to_dev(kb), to_dev(vb)
        kd[:, :, 100:] = float("nan")
        vd[:, :, 100:] = float("nan")
        kd[1, :, 3:] = float("inf")
        vd[1, :, 3:] = float("nan")
        cache.load_prefix(0, kd, vd, max_seq)
        qb = gen.gen_q(5, 0, b, h, d)
        out = torch.empty((b, h, d), dtype=torch.bfloat16, device="cuda")
        cache.decode_attention(0, to_dev(qb), out, lens)
        ref = oracle.OracleCache([0], h, g, d, b, max_seq)
        ref.load_prefix(0, gen.bf16_bits_to_f64(kb), gen.bf16_bits_to_f64(vb), max_seq)
        expect = ref.decode(0, gen.bf16_bits_to_f64(qb), lens)
        got = from_dev(out)
        assert np.isfinite(got).all()
        mx, mean = errors(got, expect)
        assert mx <= 2e-2 and mean <= 2e-3
        cache.sync_status()


@pytest.mark.parametrize("d", [64, 128])
def test_merge_of_hundreds_of_pieces(d):
    # one segment of 313 tiles over 313 CTAs: the decode launch writes partials only and the
    # combine kernel merges them
    run_small_case([0], 16, 1, d, 1, [20000], 20000, seed=15,
                   options={"grid": 600, "tile_tokens": 64}, expect={"last_deferred_merge": 1})
    run_small_case([0], 16, 1, d, 1, [20000], 20000, seed=16,
                   options={"grid": 600, "tile_tokens": 64}, fused=True,
                   expect={"last_deferred_merge": 1})


def test_long_single_segments_default_launch():
    # batch 2 x 2 KV heads of 30000 positions: four segments over the whole GPU
    run_small_case([0, 0], 8, 2, 64, 2, [30000, 29999], 30000, seed=19, fused=True,
                   expect={"last_deferred_merge": 1})


def test_few_pieces_merge_inline():
    run_small_case([0], 8, 2, 64, 4, [700, 1, 129, 1000], 1024, seed=20,
                   options={"grid": 3, "tile_tokens": 64}, expect={"last_deferred_merge": 0})


@pytest.mark.parametrize("b,L,tile,k,want_tile", [(64, 2048, 256, 2, 256), (64, 2048, 0, 4, 128),
                                                   (32, 2048, 0, 4, 128), (64, 256, 64, 4, 64)])
@pytest.mark.parametrize("fused", [False, True])
def test_cluster_merge(b, L, tile, k, want_tile, fused):
    # One length for every sequence, layer calls one by one.  64 segments of 8 tiles of 256: 2-CTA
    # clusters keep the one-wave makespan; by default 64 segments of 16 tiles of 128 (two CTAs per
    # SM): 4-CTA clusters; 32 such segments: 4-CTA clusters; 64 segments of 4 tiles of 64: 4-CTA
    # clusters.  The pieces of a segment are merged through DSMEM.
    opts = {"tile_tokens": tile} if tile else None
    run_small_case([0, 0, 2], 12, 1, 64, b, [L] * b, L, seed=17, fused=fused, options=opts,
                   expect={"last_cluster_k": k, "last_tile_tokens": want_tile})


def test_cluster_mode_off_matches():
    run_small_case([0, 0], 12, 1, 64, 64, [2048] * 64, 2048, seed=18,
                   options={"cluster": 0}, expect={"last_cluster_k": 0})


@pytest.mark.parametrize("k", [2, 4])
def test_cluster_size_forced(k):
    # The "cluster" option may name the cluster size: 2-CTA clusters of 8 tiles of 128 each (half
    # the CTAs of the default shape), or 4-CTA clusters.
    run_small_case([0, 0, 2], 12, 1, 64, 64, [2048] * 64, 2048, seed=21,
                   options={"cluster": k}, expect={"last_cluster_k": k, "last_tile_tokens": 128})


def test_cluster_rule_keeps_a_streaming_grid():
    # One long segment on the two-CTA-per-SM tile: a cluster of its pieces would be a grid of a
    # few CTAs, so the stream-K split over the SMs (and the separate merge) is kept.
    run_small_case([0, 0], 8, 1, 64, 1, [8192], 8192, seed=22, options={"tile_tokens": 128},
                   expect={"last_cluster_k": 0, "last_deferred_merge": 1})


@pytest.mark.parametrize("d,tile,tc", [(64, 64, 0), (64, 128, 0), (64, 256, 0), (128, 64, 0),
                                       (128, 128, 0), (64, 128, 1), (64, 256, 1), (128, 128, 1)])
@pytest.mark.parametrize("pieces,G,deferred", [
    (5, 3, 0), (7, 3, 0), (9, 3, 1),
    (7, 512, 0), (3, 513, 0), (4, 513, 1), (7, 513, 1), (3, 16, 0), (4, 16, 1),
])
def test_merge_of_few_pieces(d, tile, tc, pieces, G, deferred):
    # One long segment a KV head over `pieces` CTAs: where a segment can meet at most 8 CTAs (4 for
    # records of more than 512 floats) its records are merged by the last finisher, else by the merge
    # launch (runs of 2 tiles: a segment of 2 k tiles meets k CTAs, and the bound for runs that start
    # anywhere is k + 1).  G of 512 and 513: the largest group of the 8-record bound, one more.
    if G >= 512:
        G = 512 // d + G - 512
    nt = 2 * pieces
    run_small_case([0], 2 * G, 2, d, 1, [nt * tile - 5], nt * tile, seed=31, fused=True,
                   options={"grid": 2 * pieces, "tile_tokens": tile, "cluster": 0, "tc": tc},
                   expect={"last_deferred_merge": deferred, "last_tc": tc})


@pytest.mark.parametrize("d,tile", [(64, 64), (64, 128), (64, 256), (128, 64), (128, 128)])
@pytest.mark.parametrize("h,g", [(16, 1), (4, 4)])
def test_many_pieces_a_cta(d, tile, h, g):
    # Few CTAs, many short segments: every consumer warp hands its sums to the epilogue warp and
    # goes on, a piece a tile or two, whole segments and cut ones, groups of 16 heads and of one.
    lens = [1 + (i * 53) % (2 * tile) for i in range(37)]
    run_small_case([0, 0], h, g, d, len(lens), lens, 2 * tile, seed=32, fused=True,
                   options={"grid": 3, "tile_tokens": tile})


@pytest.mark.parametrize("d,tile", [(64, 64), (64, 128), (64, 256), (128, 64), (128, 128)])
@pytest.mark.parametrize("G", [1, 2, 7, 8, 9])
def test_group_sizes_around_eight(d, tile, G):
    # Groups of at most 8 heads take the kernel that holds them as the MMAs' 8 columns, larger ones
    # the 16-row kernel; whole, cut and ragged segments, new tokens in the tiles.
    lens = [1, 17, tile - 1, tile, tile + 1, 3 * tile - 7]
    run_small_case([0, 0], 2 * G, 2, d, len(lens), lens, 3 * tile, seed=33, fused=True,
                   options={"grid": 7, "tile_tokens": tile})
    run_small_case([0], 2 * G, 2, d, 2, [2 * tile, 2 * tile], 2 * tile, seed=34,
                   options={"tile_tokens": tile})


@pytest.mark.parametrize("h,g,d,b,s,options", [
    (32, 8, 128, 8, 3000, {}),                        # 6 pieces a segment at most, groups of 4
    (12, 4, 64, 64, 3000, {}),                        # groups of 3, 3 pieces
    (32, 2, 64, 12, 6000, {"tile_tokens": 128, "grid": 32}),   # the 16-row kernel
    (32, 8, 128, 8, 3000, {"tc": 1, "tile_tokens": 128}),
    (32, 2, 64, 12, 6000, {"tc": 1, "tile_tokens": 128, "grid": 32}),
])
def test_split_merges_are_reproducible(h, g, d, b, s, options):
    # A cut segment is merged by whichever CTA finishes it last, in its epilogue warp or, if the
    # piece is the CTA's last, by all its warps: the same bits every time.
    import torch

    import paper_2406_09297_gb300 as mlkv
    lens = np.array([1 + (i * 977) % s for i in range(b - 1)] + [s], dtype=np.int32)
    gen_ = torch.Generator(device="cuda").manual_seed(35)
    k, v = (torch.randn((b, g, s, d), device="cuda", generator=gen_).bfloat16() for _ in range(2))
    q = torch.randn((b, h, d), device="cuda", generator=gen_).bfloat16()
    with mlkv.MLKVCache(1, h, d, [0], g, b, s) as cache:
        for key, value in options.items():
            cache.set_option(key, value)
        cache.load_prefix(0, k, v, s)
        outs = [torch.empty_like(q) for _ in range(64)]
        for out in outs:
            cache.decode_attention(0, q, out, lens)
        torch.cuda.synchronize()
        assert cache.get_option("last_deferred_merge") == 0
        assert cache.get_option("last_tc") == options.get("tc", 0)
        for out in outs[1:]:
            assert torch.equal(out.view(torch.int16), outs[0].view(torch.int16))
        cache.sync_status()


@pytest.mark.parametrize("h", [8, 12, 16])
@pytest.mark.parametrize("tile", [64, 128, 256])
def test_largest_uneven_batch_keeps_its_tile(h, tile):
    # The length tables of the largest batch fit beside every variant's shared memory.
    b = 1024
    lens = [1 + (i * 37) % 270 for i in range(b)]
    run_small_case([0], h, 1, 64, b, lens, 270, seed=36, fused=True,
                   options={"tile_tokens": tile}, expect={"last_tile_tokens": tile})
