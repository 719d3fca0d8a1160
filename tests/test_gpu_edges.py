"""The prefill, merge, decode and copy kernels' forms at the sizes where one
gives way to the next: one-q-tile launches of a few key tiles, pairs whose
q-tiles end at different key tiles (with V's producer apart or not), split
merges around their batch of splits and their block shapes, persistent pieces of
one or two q-tiles, the plans taken by default (small workspaces too), decode
merges of one and of many chunks and the decode weights' parts, NaN and infinite
inputs, rounds against their calls made one by one, and appends, crops and
copy-on-write around the limits of their parameter blocks.  Attention is held
to the gate of tests/parity.py against the fp64 oracle; everything that moves
bytes is compared exactly."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import Pair, assert_close, dev, requires_cuda
from test_gpu_fork import _check_pools

pytestmark = [pytest.mark.gpu, requires_cuda]


def _batch(d, hq, hkv, ps, lens, nqs, options, seed):
    """One launch over sequences of `lens` keys and `nqs` queries against the oracle; returns the plan."""
    npg = sum(-(-n // ps) for n in lens) + 4
    pair = Pair(1, hkv, d, ps, npg, len(lens), max(-(-n // ps) for n in lens) + 1, seed=seed)
    for key, value in options.items():
        pair.gpu.set_option(key, value)
    g = synth.rng(seed, 71)
    seqs = []
    for n in lens:
        s = pair.seq()
        pair.append(s, synth.normal_bf16(g, (1, n, hkv, d)), synth.normal_bf16(g, (1, n, hkv, d)))
        seqs.append(s)
    cu = [0] + [int(x) for x in np.cumsum(nqs)]
    q = synth.normal_bf16(g, (cu[-1], hq, d))
    out = pair.gpu.replay_attn_batch(seqs, 0, dev(q), cu)
    torch.cuda.synchronize()
    for i, s in enumerate(seqs):
        ref = oracle.replay_attention(pair.orc, s, 0, q[cu[i]:cu[i + 1]], 1 / math.sqrt(d))
        assert_close(out[cu[i]:cu[i + 1]], ref, f"d={d} ps={ps} lens={lens} nqs={nqs} {options} seq {i}")
    assert pair.gpu.device_status() == 0
    return pair.gpu.last_attn_plan()


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("split", [0, 1])
def test_one_q_tile_launches_of_few_key_tiles(kernel, d, split):
    """Every unit one q-tile, 1 to 5 key tiles (the last ragged), whole or cut into pieces of 1 to 4."""
    lens = [40, 128, 129, 256, 300, 511, 640]
    opts = {"attn_kernel": kernel, "splitkv": split}
    if split and kernel == 0:
        opts["num_splits"] = 2
    if split and kernel == 2:
        opts["attn_ctas"] = 11
    _batch(d, 8, 2, 16, lens, [32, 20, 17, 32, 31, 9, 32], opts, seed=3 + d)


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("d,ps", [(64, 8), (64, 16), (64, 32), (128, 8), (128, 64)])
def test_pairs_whose_q_tiles_end_apart(kernel, d, ps):
    """g = 16: 8 queries a q-tile, so a pair's second q-tile reaches one key tile further where the first
    ends on a tile's edge; odd q-tile counts leave a lone one; 1 to 3 key tiles exercise every ring slot."""
    _batch(d, 16, 1, ps, [128, 136, 264, 390, 1000], [16, 24, 136, 7, 100], {"attn_kernel": kernel}, seed=d + ps)
    _batch(d, 16, 1, ps, [264, 900], [136, 300], {"attn_kernel": kernel, "splitkv": 1, "attn_ctas": 7 if kernel else 0,
                                                  "num_splits": 0 if kernel else 3}, seed=d + ps + 1)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("splits", [2, 4, 5, 8, 9, 17])
@pytest.mark.parametrize("wide", [False, True])
def test_split_merge_shapes(d, splits, wide):
    """Split counts around the merge's batches (4, then 8), with few partial rows (blocks of one warp) and
    with more than 8 MB of them (a block an SM)."""
    hq, hkv = (64, 8) if wide else (8, 2)
    nqs = [130, 70, 1] if wide else [30, 5]
    lens = [2176, 900, 70] if wide else [2176, 500]
    plan = _batch(d, hq, hkv, 16, lens, nqs, {"attn_kernel": 0, "splitkv": 1, "num_splits": splits, "decode_kernel": 0},
                  seed=splits)
    assert plan[1] == -(-17 // -(-17 // splits)), plan


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("split", [0, 1])
def test_one_q_tile_units_in_rounds(d, split):
    """14 units of one q-tile on 4 persistent CTAs: rounds of whole units, then the rest whole or cut."""
    _batch(d, 8, 2, 16, [40, 128, 129, 256, 300, 511, 640], [32, 20, 17, 32, 31, 9, 32],
           {"attn_kernel": 2, "attn_ctas": 4, "splitkv": split}, seed=5 + d)


# (d, Hq, Hkv, keys, queries): the plan's kernel and whether keys are cut, on 152 SMs
DEFAULT_PLANS = [
    # one-item: pairs and lone q-tiles with key splits and in one pass, lone ones with key splits
    (64, 32, 8, [1500, 900, 2000, 700], [200, 33, 129, 60], "one_item", True),
    (128, 32, 8, [1500, 900, 2000, 700], [200, 33, 129, 60], "one_item", True),
    (64, 16, 4, [376], [72], "one_item", False),
    (128, 32, 4, [376, 231, 244, 290, 241, 275, 256, 343, 395, 320, 271, 298, 328, 223, 314, 377, 327, 332, 338, 331],
     [87, 67, 169, 144, 56, 30, 146, 72, 177, 138, 121, 32, 187, 70, 150, 170, 52, 192, 65, 111], "one_item", False),
    (64, 32, 8, [2500, 2600], [20, 20], "one_item", True),
    (128, 32, 8, [2500, 2600], [20, 20], "one_item", True),
    (64, 16, 8, [600] * 24, [40] * 24, "persistent", False),
    (128, 16, 8, [600] * 24, [40] * 24, "one_item", False),
    # persistent with cuts (each far enough from the line that 10 to 20 % more or fewer keys keep it): pairs only, pairs and
    # lone q-tiles, lone ones only
    (64, 8, 8, [2152, 1731], [1280, 1280], "persistent", True),
    (128, 32, 8, [3105, 2492], [320, 320], "persistent", True),
    (64, 8, 8, [1686, 2153], [1243, 1449], "persistent", True),
    (128, 8, 8, [1976, 2455], [1364, 1004], "persistent", True),
    (64, 32, 8, [657, 651, 703, 791, 649, 701, 855, 769, 711, 651, 801, 634, 733, 642, 757, 831, 767, 826, 754, 857],
     [23, 10, 17, 21, 18, 19, 17, 23, 21, 19, 14, 27, 32, 27, 16, 26, 21, 17, 10, 18], "persistent", True),
    (128, 16, 16, [10979, 9572, 10189, 8719, 9407], [111, 111, 111, 86, 115], "persistent", True),
    # persistent, at least two units a SM: rounds of whole units before the cut ones
    (64, 32, 4, [827, 786, 833, 1016, 1016, 1046, 782, 763, 949, 984, 878, 1035, 765, 947, 964, 760, 1032, 841, 872, 828],
     [104, 150, 148, 70, 165, 29, 153, 107, 21, 134, 81, 140, 42, 190, 174, 114, 98, 80, 84, 96], "persistent", True),
    (128, 32, 4, [1323, 1173, 1495, 1331, 1456, 1203, 1548, 1315, 1593, 1252, 1551, 1527, 1172, 1465, 1238, 1430, 1488, 1498,
                  1572, 1188],
     [186, 128, 130, 95, 47, 41, 129, 98, 70, 83, 189, 130, 72, 132, 97, 85, 112, 141, 54, 81], "persistent", True),
    # the same with lone q-tiles only
    (64, 32, 8, [747, 907, 874, 793, 864, 884, 520, 737, 909, 561, 751, 501, 715, 643, 697, 611, 749, 712, 909, 797, 652, 788,
                 520, 893, 826, 844, 514, 580, 495, 574, 810, 596, 682, 572, 861, 864, 692, 836, 899],
     [31, 26, 15, 30, 12, 10, 17, 22, 15, 24, 15, 11, 16, 9, 29, 28, 18, 11, 25, 15, 24, 5, 10, 17, 6, 6, 14, 20, 12, 24, 10,
      23, 29, 13, 31, 13, 26, 6, 8], "persistent", True),
]


@pytest.mark.parametrize("d,hq,hkv,lens,nqs,kind,cut", DEFAULT_PLANS)
def test_default_plans_of_mixed_launches(d, hq, hkv, lens, nqs, kind, cut):
    """The plan's own choice over launches of few and of many units, of pairs, lone q-tiles and both: the kernel it
    takes, with and without cut keys, and a sample of every sequence's rows against the oracle."""
    npg = sum(-(-n // 16) for n in lens) + 4
    pair = Pair(1, hkv, d, 16, npg, len(lens), max(-(-n // 16) for n in lens) + 1, seed=len(lens) + d)
    g = synth.rng(d + len(lens), 79)
    seqs = []
    for n in lens:
        s = pair.seq()
        pair.append(s, synth.normal_bf16(g, (1, n, hkv, d)), synth.normal_bf16(g, (1, n, hkv, d)))
        seqs.append(s)
    plan = pair.gpu.plan_launches(seqs, nqs, hq)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert [(x["kind"], bool(x["split"])) for x in plan] == [(kind, cut)]
        if kind == "persistent":
            p = pair.gpu.plan_persistent(seqs, nqs, hq)
            assert (p["rounds"] > 0) == (len(p["unit_tiles"]) >= 2 * 152) and (p["n_slots"] > 0) == cut
    cu = [0] + [int(x) for x in np.cumsum(nqs)]
    q = synth.normal_bf16(g, (cu[-1], hq, d))
    out = pair.gpu.replay_attn_batch(seqs, 0, dev(q), cu)
    torch.cuda.synchronize()
    for i, s in enumerate(seqs):
        rows = np.unique(np.concatenate([np.arange(0, nqs[i], 11), [nqs[i] // 2, nqs[i] - 1]]))
        ref = oracle.replay_attention(pair.orc, s, 0, q[cu[i]:cu[i + 1]], 1 / math.sqrt(d), rows=rows)
        assert_close(out[cu[i]:cu[i + 1]][torch.from_numpy(rows).cuda()], ref, f"d={d} {kind} seq {i}")
    assert pair.gpu.device_status() == 0


@pytest.mark.parametrize("d,hq,hkv", [(128, 8, 2), (64, 16, 1), (128, 32, 8)])
@pytest.mark.parametrize("chunks_per_sm", [None, 1, 64])
def test_decode_merges_of_one_and_many_chunks(d, hq, hkv, chunks_per_sm):
    """Items of 1 chunk (no merge) to 71 one-tile chunks (more than one round trip of the merge) in one launch."""
    options = {} if chunks_per_sm is None else {"decode_chunks_per_sm": chunks_per_sm}
    _batch(d, hq, hkv, 16, [100, 128, 1025, 9000, 4097], [1] * 5, options, seed=d + hq)


def test_decode_chunk_option_returns_to_its_default():
    """"decode_chunks_per_sm" set and set back to 0: the plan and the bits of a cache that never had it set."""
    hq, hkv, d, n = 32, 8, 128, 6000
    g = synth.rng(3, 77)
    k, v, q = (dev(synth.normal_bf16(g, (1, n, h, d))) for h in (hkv, hkv, hq))
    got = []
    for values in ([], [64], [64, 0]):
        pair = Pair(1, hkv, d, 16, n // 16 + 4, 1, n // 16 + 2, seed=3)
        s = pair.gpu.seq_create()
        pair.gpu.append_kv(s, k, v)
        for value in values:
            pair.gpu.set_option("decode_chunks_per_sm", value)
        out = pair.gpu.replay_attn(s, 0, q[0, :1].contiguous())
        got.append((pair.gpu.last_attn_plan(), out))
    assert got[2][0] == got[0][0] != got[1][0]
    assert torch.equal(got[2][1], got[0][1])


@pytest.mark.parametrize("n", [1, 16, 17, 40])
def test_append_and_crop_around_the_small_parameter_blocks(n):
    """n sequences appended and cropped in one call each, the first append of 8 pages a sequence: 16 sequences
    make 128 pages, and 17 leave the small blocks by both counts."""
    hkv, d, ps, L = 2, 64, 16, 2
    pair = Pair(L, hkv, d, ps, 9 * n + 8, n, 10, seed=n)
    g = synth.rng(n, 72)
    seqs = [pair.seq() for _ in range(n)]
    for lens in ([128] * n, [1 + (7 * i) % 15 for i in range(n)]):
        cu = [0] + [int(x) for x in np.cumsum(lens)]
        k, v = (synth.normal_bf16(g, (L, cu[-1], hkv, d)) for _ in range(2))
        pair.gpu.append_kv_batch(seqs, dev(k), dev(v), cu)
        for i, s in enumerate(seqs):
            pair.orc.append(s, k[:, cu[i]:cu[i + 1]], v[:, cu[i]:cu[i + 1]])
        pair.check_state(seqs)
    _check_pools(pair, L, hkv, ps, d)
    taus = [1 + (5 * i) % 40 for i in range(n)]
    pair.gpu.crop_batch(seqs, taus)
    for s, tau in zip(seqs, taus):
        pair.orc.crop(s, tau)
    pair.check_state(seqs)
    _check_pools(pair, L, hkv, ps, d)


@pytest.mark.parametrize("branches", [1, 63, 64, 65])
def test_copy_on_write_of_many_branches_in_one_append(branches):
    """Each branch of a base whose last page is half full gets its own copy of that page in one append."""
    hkv, d, ps, L, T = 2, 64, 16, 2, 40
    pair = Pair(L, hkv, d, ps, 3 + 2 * branches + 4, branches + 1, 5, seed=branches)
    g = synth.rng(branches, 73)
    base = pair.seq()
    pair.append(base, synth.normal_bf16(g, (L, T, hkv, d)), synth.normal_bf16(g, (L, T, hkv, d)))
    seqs = []
    for _ in range(branches):
        a, b = pair.gpu.seq_fork(base), pair.orc.seq_fork(base)
        assert a == b
        seqs.append(a)
    cu = list(range(0, 3 * branches + 1, 3))
    k, v = (synth.normal_bf16(g, (L, cu[-1], hkv, d)) for _ in range(2))
    pair.gpu.append_kv_batch(seqs, dev(k), dev(v), cu)
    for i, s in enumerate(seqs):
        pair.orc.append(s, k[:, cu[i]:cu[i + 1]], v[:, cu[i]:cu[i + 1]])
    pair.check_state([base] + seqs)
    _check_pools(pair, L, hkv, ps, d)


@pytest.mark.parametrize("layers,keys", [(1, (60, 90)), (1, (700, 1300)), (1, (100, 3000)), (3, (700, 1300))])
def test_rounds_equal_their_calls_one_by_one(layers, keys):
    """Decode rounds in one call, where a round's append runs beside the merge before it, against the same
    appends and attention calls made one by one: the same output bits, pages and lengths.  Items of one
    chunk (no merge), of several, and both; a fork's copy-on-write before the first append."""
    hq, hkv, d, ps, rounds = 32, 8, 128, 16, 12
    g = synth.rng(sum(keys), 74)
    base = [(synth.normal_bf16(g, (layers, n, hkv, d)), synth.normal_bf16(g, (layers, n, hkv, d))) for n in keys]
    n = len(keys) + 1
    cu = [rounds * i for i in range(n + 1)]
    K, V, Q = (dev(synth.normal_bf16(g, (layers, cu[-1], h, d))) for h in (hkv, hkv, hq))
    outs, pools = [], []
    for whole in (True, False):
        pair = Pair(layers, hkv, d, ps, sum(-(-k // ps) for k in keys) + 2 * n + 8, n, 220, seed=6)
        seqs = []
        for k, v in base:
            s = pair.seq()
            pair.append(s, k, v)
            seqs.append(s)
        seqs.append(pair.gpu.seq_fork(seqs[0]))
        out = torch.zeros((layers, cu[-1], hq, d), dtype=torch.bfloat16, device="cuda")
        if whole:
            pair.gpu.replay_rounds(seqs, [[1] * n] * rounds, cu, K, V, Q, out=out)
        else:
            for r in range(rounds):
                idx = torch.tensor([c + r for c in cu[:-1]], device="cuda")
                pair.gpu.append_kv_batch(seqs, K[:, idx].contiguous(), V[:, idx].contiguous(), list(range(n + 1)))
                for layer in range(layers):
                    out[layer, idx] = pair.gpu.replay_attn_batch(seqs, layer, Q[layer, idx].contiguous(),
                                                                 list(range(n + 1)))
        torch.cuda.synchronize()
        assert pair.gpu.device_status() == 0
        outs.append(out)
        pools.append([(x, pair.gpu.page_table(s)) for s in seqs for x in [pair.gpu.seq_info(s)]])
    assert torch.equal(outs[0], outs[1])
    assert pools[0] == pools[1]
    assert outs[0].float().abs().sum() > 0


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("hq,hkv,nq", [(8, 8, 1), (32, 8, 1), (24, 3, 1), (32, 8, 3), (32, 4, 2)])
@pytest.mark.parametrize("lens", [[12003], [9000, 4097, 1100, 300], [700] * 12])
def test_decode_error_does_not_grow_with_the_chunks(d, hq, hkv, nq, lens):
    """1 to 16 rows per kv-head: the default chunk length is as close to 64 bits as three chunks a SM are (2 % for
    what regrouped sums differ by).  Where chunks are longer the weights have two parts, and what is off is the
    output's rounding to bf16, at most 2^-9 of each value; the weights' 16 bits and the fp32 sums add less than
    2^-17 of the mean weighted |V|, some 50 |O| here and independent across keys: below 8e-5 of the output."""
    npg = sum(-(-n // 16) for n in lens) + 4
    pair = Pair(1, hkv, d, 16, npg, len(lens), max(lens) // 16 + 2, seed=d + hq)
    g = synth.rng(d + hq + nq, 75)
    seqs = []
    for n in lens:
        s = pair.seq()
        pair.append(s, synth.normal_bf16(g, (1, n, hkv, d)), synth.normal_bf16(g, (1, n, hkv, d)))
        seqs.append(s)
    cu = [nq * i for i in range(len(lens) + 1)]
    q = synth.normal_bf16(g, (cu[-1], hq, d))
    ref = np.concatenate([oracle.replay_attention(pair.orc, s, 0, q[cu[i]:cu[i + 1]], 1 / math.sqrt(d))
                          for i, s in enumerate(seqs)])
    err, splits = [], []
    for chunks_per_sm in (0, 3):
        pair.gpu.set_option("decode_chunks_per_sm", chunks_per_sm)
        out = pair.gpu.replay_attn_batch(seqs, 0, dev(q), cu)
        torch.cuda.synchronize()
        splits.append(pair.gpu.last_attn_plan()[1])
        err.append(np.linalg.norm(out.double().cpu().numpy() - ref) / np.linalg.norm(ref))
    assert pair.gpu.device_status() == 0
    assert err[0] <= 1.02 * err[1], (err, splits)
    if splits[0] < splits[1]:
        assert err[0] <= 2.0 ** -9 + 8e-5, (err, splits)


@pytest.mark.parametrize("inf_at", [11000, 5])
def test_decode_of_an_infinite_value_is_infinite(inf_at):
    """V infinite at a key whose weight is the row's largest (exactly 1 against the row's reference) and at others:
    the output is that infinity, not NaN."""
    hq, hkv, d, n = 64, 8, 128, 12000
    pair = Pair(1, hkv, d, 16, n // 16 + 4, 1, n // 16 + 2, seed=9)
    g = synth.rng(9, 78)
    k, v, q = (synth.bits_to_torch(synth.normal_bf16(g, (1, n, h, d))) for h in (hkv, hkv, hq))
    q1 = q[0, :1].clone()
    k[0, inf_at, 2] = q1[0, 16:24].float().sum(0).to(torch.bfloat16)  # the key nearest to the head group's queries
    v[0, inf_at, 2, 7] = float("inf")
    s = pair.gpu.seq_create()
    pair.gpu.append_kv(s, k.cuda(), v.cuda())
    out = pair.gpu.replay_attn(s, 0, q1.cuda())
    assert torch.isposinf(out[0, 16:24, 7]).all()
    out[0, 16:24, 7] = 0
    assert torch.isfinite(out).all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("nq", [1, 40, 130])
@pytest.mark.parametrize("options", [{}, {"attn_kernel": 0, "splitkv": 0}, {"attn_kernel": 0, "num_splits": 3, "splitkv": 1},
                                     {"attn_kernel": 0, "num_splits": 20, "splitkv": 1}, {"attn_kernel": 2, "attn_ctas": 9},
                                     {"attn_kernel": 2, "attn_ctas": 60}])
@pytest.mark.parametrize("where", ["one", "most"])
def test_a_nan_key_reaches_every_output_that_attends_it(d, nq, options, where):
    """A NaN among one kv-head's keys makes that head's outputs NaN, whatever parts the keys are cut into: one
    part with the NaN, or a NaN in each but the last (more such parts than a merge takes at once).  The other
    heads are not touched."""
    hq, hkv, n = 8, 2, 2600
    pair = Pair(1, hkv, d, 16, n // 16 + 4, 1, n // 16 + 2, seed=d + nq)
    for key, value in options.items():
        pair.gpu.set_option(key, value)
    g = synth.rng(d + nq, 76)
    s = pair.seq()
    k, v = (synth.normal_bf16(g, (1, n, hkv, d)) for _ in range(2))
    q = synth.normal_bf16(g, (nq, hq, d))
    pair.orc.append(s, k, v)
    ref = oracle.replay_attention(pair.orc, s, 0, q, 1 / math.sqrt(d))
    bad = k.copy()
    bad[0, [5] if where == "one" else list(range(3, 2400, 128)), 1, 7] = 0x7FC0
    pair.gpu.append_kv(s, dev(bad), dev(v))
    out = pair.gpu.replay_attn(s, 0, dev(q))
    torch.cuda.synchronize()
    assert pair.gpu.device_status() == 0
    assert_close(out[:, :4], ref[:, :4], f"{options}")
    assert torch.isnan(out[:, 4:]).all(), (options, pair.gpu.last_attn_plan())


@pytest.mark.parametrize("keys", [(700, 1300), (100, 3000)])
def test_rounds_with_out_over_the_next_keys(keys):
    """Decode rounds whose out row j is K's row j + 1 (one buffer): a round's output is the next round's key, so its
    append must not run beside the merge that writes it.  Against the same calls made one by one."""
    h, d, ps, rounds = 8, 128, 16, 24
    g = synth.rng(sum(keys), 80)
    base = [(synth.normal_bf16(g, (1, n, h, d)), synth.normal_bf16(g, (1, n, h, d))) for n in keys]
    n = len(keys)
    cu = [rounds * i for i in range(n + 1)]
    first, V, Q = (dev(synth.normal_bf16(g, (1, cu[-1] + 1, h, d))) for _ in range(3))
    V, Q = V[:, :-1].contiguous(), Q[:, :-1].contiguous()
    got = []
    for whole in (True, False):
        pair = Pair(1, h, d, ps, sum(-(-k // ps) for k in keys) + 2 * n + 8, n, 220, seed=7)
        seqs = []
        for k, v in base:
            s = pair.seq()
            pair.append(s, k, v)
            seqs.append(s)
        buf = first.clone()
        K, out = buf[:, :-1], buf[:, 1:]
        if whole:
            pair.gpu.replay_rounds(seqs, [[1] * n] * rounds, cu, K, V, Q, out=out)
        else:
            for r in range(rounds):
                idx = torch.tensor([c + r for c in cu[:-1]], device="cuda")
                pair.gpu.append_kv_batch(seqs, K[:, idx].contiguous(), V[:, idx].contiguous(), list(range(n + 1)))
                out[0, idx] = pair.gpu.replay_attn_batch(seqs, 0, Q[0, idx].contiguous(), list(range(n + 1)))
        torch.cuda.synchronize()
        assert pair.gpu.device_status() == 0
        got.append(buf)
    assert torch.equal(got[0], got[1])
    assert not torch.equal(got[0], first)


@pytest.mark.parametrize("d,lens,nqs,hq,ws", [(64, [8192] * 3, [20] * 3, 64, 1 << 20), (128, [2490, 1746], [256, 384], 32, 4 << 20),
                                              (128, [2490, 1746], [256, 384], 32, 24 << 20)])
def test_default_plans_with_a_small_workspace(d, lens, nqs, hq, ws):
    """The default plan where the workspace holds none or some of the parts that cuts would need."""
    hkv = 8
    npg = sum(-(-n // 16) for n in lens) + 4
    pair = Pair(1, hkv, d, 16, npg, len(lens), max(lens) // 16 + 2, seed=d, pe_kwargs={"workspace_bytes": ws})
    g = synth.rng(d + ws, 81)
    seqs = []
    for n in lens:
        s = pair.seq()
        pair.append(s, synth.normal_bf16(g, (1, n, hkv, d)), synth.normal_bf16(g, (1, n, hkv, d)))
        seqs.append(s)
    cu = [0] + [int(x) for x in np.cumsum(nqs)]
    q = synth.normal_bf16(g, (cu[-1], hq, d))
    out = pair.gpu.replay_attn_batch(seqs, 0, dev(q), cu)
    torch.cuda.synchronize()
    for i, s in enumerate(seqs):
        rows = np.arange(0, nqs[i], 7)
        ref = oracle.replay_attention(pair.orc, s, 0, q[cu[i]:cu[i + 1]], 1 / math.sqrt(d), rows=rows)
        assert_close(out[cu[i]:cu[i + 1]][torch.from_numpy(rows).cuda()], ref, f"ws={ws} seq {i}")
    assert pair.gpu.device_status() == 0
