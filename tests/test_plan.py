"""The decode planner on the CPU (uc_attend_plan with an explicit CTA-slot
count, so no device is touched): how a decode-shaped call is split into
split-K work items (App. E), hand-worked for the long-context shapes and
checked for its invariants over seeded random segment mixes."""
import ctypes as C

import numpy as np
import pytest

from paper_2609_32831_gb300 import _lib, api

SLOTS = 3 * 152          # single-tile calls: three CTAs on each of 152 SMs


def _seg(kind, bits, kept, hkv=4):
    s = _lib.UcSegment()
    s.kind, s.bits, s.batch, s.n_kv_heads, s.head_dim = kind, bits, len(kept), hkv, 128
    s.cap = max(max(kept), 1)
    for b, n in enumerate(kept):
        s.n_kept_host[b] = n
    return s


def _tiles(kind, bits, n):
    """(heavy tiles, tail tile) of a segment holding n tokens: 64-row bf16
    tiles, or packed tiles of 8 (int2) / 4 (int4) groups of 32 plus a bf16
    tail of n mod 32 tokens."""
    if kind in (_lib.KIND_FULL, _lib.KIND_EVICT):
        return -(-n // 64), 0
    g = n // 32
    per = 8 if bits == 2 else 4
    return -(-g // per), int(n % 32 > 0)


def test_long_context_32k_hand_worked():
    # batch 16: 3276 text + 29492 image tokens, both int2, 128 generated bf16
    text = _seg(_lib.KIND_QUANT, 2, [3276] * 16)
    vit = _seg(_lib.KIND_QUANT, 2, [29492] * 16)
    gen = _seg(_lib.KIND_EVICT, 16, [128] * 16)
    p = api.attend_plan([text, vit, gen], 28, 1, SLOTS)
    # heavy tiles: text ceil(102 / 8) = 13, image ceil(921 / 8) = 116 (24 KB
    # each); generated 2 bf16 tiles (64 KB) < half of the 3.2 MB / 7 average
    # item -> light. 7 heavy items fill 64 * 7 = 448 of 456 slots (>= 90 %);
    # split so the largest item is smallest: text 1 (13 tiles), image 6
    # (20 tiles; 5 would give 24). Light: both int2 tails and the bf16 segment.
    assert _tiles(_lib.KIND_QUANT, 2, 3276) == (13, 1)
    assert _tiles(_lib.KIND_QUANT, 2, 29492) == (116, 1)
    assert p["n_heavy"] == 7 and p["n_light"] == 3 and p["items_per_bh"] == 10
    assert p["n_chunks"] == [2, 7, 1]
    assert p["light"] == [False, False, True]
    assert p["grid"] == SLOTS and not p["merge_kernel"]


def test_understanding_8k_hand_worked():
    # batch 8 x 4 KV heads = 32 (sequence, KV head) pairs: 512 text bf16 rows
    # (8 tiles of 64 rows, 32 KB each), 2150 kept image tokens int4 (67
    # groups: 17 tiles of 4 groups, 20 KB each, + a 6-token tail), 512
    # generated tokens int2 (16 groups: 2 tiles of 8 groups, 24 KB each).
    text = _seg(_lib.KIND_FULL, 16, [512] * 8)
    vit = _seg(_lib.KIND_EVICT_QUANT, 4, [2150] * 8)
    gen = _seg(_lib.KIND_QUANT, 2, [512] * 8)
    assert _tiles(_lib.KIND_FULL, 16, 512) == (8, 0)
    assert _tiles(_lib.KIND_EVICT_QUANT, 4, 2150) == (17, 1)
    assert _tiles(_lib.KIND_QUANT, 2, 512) == (2, 0)
    p = api.attend_plan([text, vit, gen], 28, 1, SLOTS)
    # 13 heavy items would fill 416 of 456 slots (>= 90 %), but with the two
    # packed tails that is 15 > 14 items, and 12 still fill 384 (84 % >= 80
    # %). Largest item smallest, one item at a time: image 6 items (3 tiles, 60
    # KB), text 5 (2 tiles, 64 KB), generated 1 (48 KB). The fifth text item
    # leaves the largest text item at 2 tiles, so it is dropped: text 4, image
    # 6 + tail, generated 1 + tail (empty here) = 13 items, 11 of them heavy.
    assert p["n_chunks"] == [4, 7, 2]
    assert p["n_heavy"] == 11 and p["n_light"] == 2 and p["items_per_bh"] == 13
    assert p["grid"] == 13 * 32 and not p["merge_kernel"]


def test_no_item_leaves_a_segments_largest_item_as_it_was():
    # in a plan of few items a segment of 8 tiles takes 4 items of 2 rather
    # than 5 of 1-2, whatever count the slot fill asked for
    for tiles, kind, bits, n in [(8, _lib.KIND_FULL, 16, 512), (17, _lib.KIND_QUANT, 4, 2144)]:
        seg = _seg(kind, bits, [n] * 2, hkv=1)
        for slots in (4, 6, 10, 12, 20, 30, 40):
            p = api.attend_plan([seg], 7, 1, slots)
            heavy = p["n_chunks"][0] - (1 if kind == _lib.KIND_QUANT else 0)
            per = -(-tiles // heavy)
            assert heavy == -(-tiles // per), (tiles, slots, heavy)


def test_long_context_128k_uses_the_merge_kernel():
    # batch 2: 8 (sequence, KV head) pairs need ~56 items each to fill 456 slots
    text = _seg(_lib.KIND_QUANT, 2, [13107] * 2)
    vit = _seg(_lib.KIND_QUANT, 2, [117965] * 2)
    p = api.attend_plan([text, vit], 28, 1, SLOTS)
    assert p["n_heavy"] * 8 >= 0.9 * SLOTS and p["n_heavy"] <= 56
    assert p["items_per_bh"] == p["n_heavy"] + 2 > 32
    assert p["merge_kernel"] and p["light"] == [False, False]


def test_a_short_segment_keeps_its_own_item_when_comparable():
    # two halves of equal size: neither is light, the items split evenly
    a = _seg(_lib.KIND_QUANT, 4, [8192] * 16)
    b = _seg(_lib.KIND_QUANT, 4, [8192] * 16)
    p = api.attend_plan([a, b], 28, 1, SLOTS)
    assert p["light"] == [False, False]
    assert abs(p["n_chunks"][0] - p["n_chunks"][1]) <= 1


def test_empty_segment_is_one_light_item():
    full = _seg(_lib.KIND_EVICT, 16, [4000] * 4)
    empty = _seg(_lib.KIND_EVICT, 16, [0] * 4)
    p = api.attend_plan([full, empty], 28, 1, SLOTS)
    assert p["light"] == [False, True] and p["n_chunks"][1] == 1


@pytest.mark.parametrize("seed", range(40))
def test_plan_invariants_random_mixes(seed):
    rng = np.random.default_rng(seed)
    nseg = int(rng.integers(1, 9))
    B = int(rng.choice([1, 2, 3, 8, 16, 64]))
    hkv = int(rng.choice([1, 2, 4, 8]))
    kinds = [int(k) for k in rng.integers(0, 4, nseg)]
    segs = []
    for k in kinds:
        bits = 16 if k in (_lib.KIND_FULL, _lib.KIND_EVICT) else int(rng.choice([2, 4]))
        top = int(rng.choice([1, 40, 700, 9000, 60000]))
        segs.append(_seg(k, bits, [int(x) for x in rng.integers(0, top + 1, B)], hkv))
    T = int(rng.integers(1, 9))
    slots = int(rng.choice([152, 456]))
    p = api.attend_plan(segs, 7 * hkv, T, slots)
    nbh = B * hkv
    assert 1 <= p["items_per_bh"] <= 64
    assert p["n_heavy"] + p["n_light"] == p["items_per_bh"] == sum(p["n_chunks"])
    assert p["n_heavy"] <= 56 and p["n_light"] <= 2 * nseg
    assert all(c >= 1 for c in p["n_chunks"])
    assert p["grid"] == min(p["items_per_bh"] * nbh, slots)
    assert p["merge_kernel"] == (p["items_per_bh"] > 32)
    for s, seg in zip(range(nseg), segs):
        packed = seg.kind in (_lib.KIND_QUANT, _lib.KIND_EVICT_QUANT)
        if p["light"][s]:
            # a light segment is one item, or its packed tiles and its tail
            assert p["n_chunks"][s] <= (2 if packed else 1)
        else:
            # a heavy packed segment ends with its (light) tail item
            assert p["n_chunks"][s] >= (2 if packed else 1)
            # and, in a plan of few items, takes no item that leaves its
            # largest item as large
            tiles = _tiles(seg.kind, seg.bits, max(seg.n_kept_host[b] for b in range(B)))[0]
            hc = p["n_chunks"][s] - (1 if packed else 0)
            per = -(-tiles // hc)
            if not p["merge_kernel"]:
                assert hc == -(-tiles // per)


# cluster CTAs, merge width of the short-call mixes on 456 slots
CLUSTERS = {"one_token": (1, 0), "tails_only": (4, 0), "eight_segments": (14, 0), "shared_light_rank": (12, 0),
            "one_long_pair": (0, 32), "ragged": (16, 0), "pairs_64": (6, 0), "pairs_512": (0, 128)}


def test_short_calls_and_their_clusters():
    """One rank per heavy item and one for every light item, or a single one
    for all of them where a cluster of more would not fit often enough; the
    GPU tests run the same mixes."""
    from tests.test_gpu_kernels import CLUSTER_MIXES
    assert set(CLUSTERS) == set(CLUSTER_MIXES)
    kind_of = api.KIND_NAMES
    for mix, (B, hkv, _, kinds, keeps, bits) in CLUSTER_MIXES.items():
        segs = [_seg(kind_of[k], bt, kp if hasattr(kp, "__len__") else [kp] * B, hkv)
                for k, kp, bt in zip(kinds, keeps, bits)]
        p = api.attend_plan(segs, 7 * hkv, 1, SLOTS)
        assert (p["cluster"], p["merge_width"]) == CLUSTERS[mix], mix
        if p["cluster"]:
            assert p["cluster"] - p["n_heavy"] in (0 if p["n_light"] == 0 else 1, p["n_light"]), mix
            assert p["ctas"] == p["cluster"] * B * hkv <= SLOTS and p["stages"] == 2
        else:
            assert p["ctas"] == p["grid"]
    # two light items, one rank for both
    B, hkv, _, kinds, keeps, bits = CLUSTER_MIXES["shared_light_rank"]
    p = api.attend_plan([_seg(kind_of[k], bt, [kp] * B, hkv) for k, kp, bt in zip(kinds, keeps, bits)], 28, 1, SLOTS)
    assert p["n_light"] == 2 and p["cluster"] == p["n_heavy"] + 1


def test_launches_of_the_hand_worked_calls():
    """The 32K layer walks its items as a queue and merges 64 pairs by CTAs of
    32 channels; the 8K layer's 32 pairs are clusters of 12."""
    seg32 = [_seg(_lib.KIND_QUANT, 2, [3276] * 16), _seg(_lib.KIND_QUANT, 2, [29492] * 16),
             _seg(_lib.KIND_EVICT, 16, [128] * 16)]
    p = api.attend_plan(seg32, 28, 1, SLOTS)
    assert (p["cluster"], p["ctas"], p["stages"], p["merge_width"]) == (0, SLOTS, 2, 32)
    seg8 = [_seg(_lib.KIND_FULL, 16, [512] * 8), _seg(_lib.KIND_EVICT_QUANT, 4, [2150] * 8),
            _seg(_lib.KIND_QUANT, 2, [512] * 8)]
    p = api.attend_plan(seg8, 28, 1, SLOTS)
    assert (p["cluster"], p["ctas"], p["merge_width"]) == (12, 12 * 32, 0)
    # four query tokens: four row blocks of each pair, three ring slots only
    # where the CTAs are no more than the SMs
    p = api.attend_plan([_seg(_lib.KIND_FULL, 16, [43000])], 28, 4, 2 * 152)
    assert (p["cluster"], p["stages"]) == (0, 3) and p["ctas"] <= 152
    p = api.attend_plan(seg8, 28, 4, 2 * 152)
    assert (p["cluster"], p["stages"], p["merge_width"]) == (0, 2, 64)   # 128 (pair, row block)s


def test_plan_rejects_bad_calls():
    h = _lib.lib()
    seg = _seg(_lib.KIND_QUANT, 2, [64])
    arr = (C.POINTER(_lib.UcSegment) * 1)(C.pointer(seg))
    info = _lib.UcAttendPlanInfo()
    n0 = h.uc_launch_count()
    assert h.uc_attend_plan(None, 1, 28, 1, SLOTS, C.byref(info)) == _lib.UC_ERR_ARG
    assert h.uc_attend_plan(C.cast(arr, C.c_void_p), 1, 28, 9, SLOTS, C.byref(info)) == _lib.UC_ERR_SHAPE
    assert h.uc_attend_plan(C.cast(arr, C.c_void_p), 1, 30, 1, SLOTS, C.byref(info)) == _lib.UC_ERR_SHAPE
    seg.bits = 3
    assert h.uc_attend_plan(C.cast(arr, C.c_void_p), 1, 28, 1, SLOTS, C.byref(info)) == _lib.UC_ERR_SHAPE
    run = _lib.UcAttendLaunchInfo()
    assert h.uc_attend_launch(None, 1, 28, 1, SLOTS, C.byref(run)) == _lib.UC_ERR_ARG
    assert h.uc_attend_launch(C.cast(arr, C.c_void_p), 1, 28, 1, SLOTS, C.byref(run)) == _lib.UC_ERR_SHAPE
    assert h.uc_launch_count() == n0
