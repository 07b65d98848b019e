"""How a call is cut into work, from the functions that decide it: which kernel and form a shape takes, and that every piece of
the product belongs to exactly one task."""
import ctypes
import random

import numpy as np
import pytest

import paper_2406_13868_b200 as m

FEW, PAIRS, GROUP = 0, 1, 2
TWO, FULL, FLEX = 0, 1, 2
i64 = ctypes.c_int64


class Plan(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("kernel", "token_tile", "ksplit", "cluster", "ctas", "tasks", "form", "alternate", "doubles", "halves",
                                              "rounds", "tail_items")]


def machine(sms, clusters):
    return ctypes.c_int(sms), (ctypes.c_int * 5)(0, 0, *clusters)


def linear_plan(M, N, K, cfg, on, workspace=0):
    m.build()
    plan, cap = Plan(), 1 << 16
    tasks = np.zeros((cap, 5), np.int32)
    st = m.lib().sdq_diag_linear_plan(i64(M), i64(N), i64(K), ctypes.byref(cfg), workspace, *on, ctypes.byref(plan), tasks.ctypes.data_as(ctypes.c_void_p), i64(cap))
    assert st == 0 and plan.tasks <= cap
    return plan, tasks[:plan.tasks]


def group_plan(M, shapes, on):
    m.build()
    plan, cap, n = Plan(), 1 << 16, len(shapes)
    segs = np.zeros((cap, 5), np.int32)
    st = m.lib().sdq_diag_group_plan(n, i64(M), (i64 * n)(*[s[0] for s in shapes]), (i64 * n)(*[s[1] for s in shapes]), *on, ctypes.byref(plan),
                                     segs.ctypes.data_as(ctypes.c_void_p), i64(cap))
    assert st == 0 and plan.tasks <= cap
    return plan, segs[:plan.tasks]


class Rings(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("slots", "slot_bytes", "out_slots", "out_slot_bytes", "bytes")]


def linear_rings(M, N, K, cfg, on):
    m.build()
    r = Rings()
    assert m.lib().sdq_diag_linear_rings(i64(M), i64(N), i64(K), ctypes.byref(cfg), *on, ctypes.byref(r)) == 0
    return r


def cover_pairs(plan, tasks, M, N):
    units, groups = -(-N // 256), -(-M // 32)
    seen = np.zeros((units, groups), np.int32)
    for _, row, rows, g0, g1 in tasks:
        assert rows in (1, 2) and g0 < g1 and 32 * (g1 - g0) <= plan.token_tile
        assert row + rows <= units and g1 <= groups
        seen[row:row + rows, g0:g1] += 1
    assert (seen == 1).all()
    if plan.form != TWO:
        assert plan.doubles == plan.halves == 0
    if plan.ksplit > 1:                                   # one task per cluster, all clusters at once
        assert plan.form == FLEX and plan.ctas == plan.cluster * plan.tasks and plan.cluster == 2 * plan.ksplit
        assert plan.alternate or plan.ksplit == 2         # tiles too wide to alternate are shared by two pairs at most


def cover_group(plan, segs, shapes):
    seen = [np.zeros((n // 128, k // 256), np.int32) for n, k in shapes]
    for layer, row, rows, b, e in segs:
        assert rows == 1 and b < e
        seen[layer][row, b:e] += 1
    assert all((s == 1).all() for s in seen)
    # a CTA's item may be shared only at the end of its work, by neighbours of one cluster
    assert plan.cluster in (1, 2, 4) and plan.ctas % plan.cluster == 0 and plan.ksplit * plan.tail_items == plan.cluster


@pytest.mark.parametrize("sms,clusters", [(148, (36, 24, 16)), (148, (0, 0, 0)), (132, (33, 16, 16)), (20, (5, 3, 2))])
def test_every_piece_of_a_product_belongs_to_one_task(sms, clusters):
    on, rng = machine(sms, clusters), random.Random(sms)
    kinds = set()
    for _ in range(250):
        M, N, K = (int(round(2 ** rng.uniform(0, b))) for b in (13, 7.2, 6.2))
        N, K = 128 * N, 256 * K
        cfg = rng.choice([m.Config(rng.randint(0, 2), m.GRAN_PAIR, 64), m.Config(1, m.GRAN_PAIR, 32, m.SCALE_UE4M3), m.Config(1, m.GRAN_DENSE, 32)])
        plan, tasks = linear_plan(M, N, K, cfg, on)
        if plan.kernel == PAIRS:
            cover_pairs(plan, tasks, M, N)
            assert plan.ksplit <= K // 256 and plan.ctas <= sms
            if plan.ksplit > 1:
                assert plan.tasks <= clusters[plan.ksplit - 2]
        elif plan.kernel == GROUP:
            cover_group(plan, tasks, [(N, K)])
        else:
            assert M <= 128 and 1 <= plan.ksplit <= 8 and plan.ksplit <= K // 256
        assert M <= 128 or plan.kernel == PAIRS
        kinds.add((plan.kernel, plan.form))
    assert {(PAIRS, TWO), (PAIRS, FLEX), (GROUP, 0)} <= kinds
    for _ in range(100):
        shapes = [(128 * rng.randint(1, 90), 256 * rng.randint(4, 44)) for _ in range(rng.randint(1, 12))]
        plan, segs = group_plan(rng.randint(1, 32), shapes, on)
        cover_group(plan, segs, shapes)


B200 = (148, (33, 22, 15))
PAIR, B32, UE, DENSE, NONE = m.Config(1, 0, 64, 0), m.Config(2, 0, 32, 1), m.Config(1, 0, 32, 2), m.Config(1, m.GRAN_DENSE, 32, 0), m.Config(0)
# the shapes of the parity tests of each form -> what runs there (`split`: K is)
FORMS = [
    (3371, 2560, 2048, PAIR, dict(kernel=PAIRS, form=FULL, split=False)),
    (3371, 2688, 2048, PAIR, dict(kernel=PAIRS, form=TWO, halves=True)),
    (5001, 1280, 2048, PAIR, dict(kernel=PAIRS, form=TWO, halves=False)),
    (2901, 3200, 2048, B32, dict(kernel=PAIRS, form=TWO)),
    (4001, 2304, 2048, UE, dict(kernel=PAIRS, form=FULL)),
    (4001, 1664, 2048, DENSE, dict(kernel=PAIRS, form=FLEX, alternate=True, split=False)),
    (4096, 11008, 4096, DENSE, dict(kernel=PAIRS, form=FULL)),          # dense inliers, several rounds: one-unit tasks are faster
    (4096, 4096, 16384, DENSE, dict(kernel=PAIRS, form=FULL)),
    (1500, 16384, 4096, m.Config(1, m.gran_keep(7), 32), dict(kernel=PAIRS, form=FULL)),
    (1500, 4096, 11008, DENSE, dict(kernel=PAIRS, form=TWO)),           # ... one round: two-unit tasks are
    (2048, 2560, 1280, DENSE, dict(kernel=PAIRS, form=TWO)),
    (300, 384, 2048, UE, dict(kernel=PAIRS, form=FLEX, split=True)),
    (200, 384, 1536, DENSE, dict(kernel=PAIRS, form=FLEX, split=True)),
    (100, 4096, 2048, PAIR, dict(kernel=PAIRS, form=FLEX, split=True)),
    (64, 2176, 4096, m.Config(2), dict(kernel=FEW, split=True)),
    (130, 128, 256, NONE, dict(kernel=PAIRS, form=FLEX, split=False)),
    (3371, 2688, 2048, UE, dict(kernel=PAIRS, form=TWO)),
    (497, 3968, 4096, PAIR, dict(kernel=PAIRS, form=FLEX, split=True, ksplit=2, alternate=False, token_tile=256)),
    (450, 3840, 4352, UE, dict(kernel=PAIRS, form=FLEX, split=True, ksplit=2, alternate=False, token_tile=256)),
    (512, 4096, 4096, DENSE, dict(kernel=PAIRS, form=FLEX, split=True, ksplit=2, alternate=False, token_tile=256)),
    (213, 6656, 5632, DENSE, dict(kernel=PAIRS, form=FLEX, split=True, ksplit=2, alternate=False, token_tile=224)),
    (220, 5120, 5120, UE, dict(kernel=PAIRS, form=FLEX, split=True, ksplit=2, alternate=False, token_tile=224)),
    (1, 4096, 4096, PAIR, dict(kernel=GROUP, split=True, rounds=False)),
    (17, 4224, 4096, PAIR, dict(kernel=GROUP, split=True, rounds=False)),
    (5, 8192, 8192, PAIR, dict(kernel=GROUP, split=True, rounds=False)),
    (3, 19072, 4096, PAIR, dict(kernel=GROUP, split=True, rounds=True)),
    (32, 8448, 2048, PAIR, dict(kernel=GROUP, split=False, rounds=False)),
    (9, 16640, 1024, NONE, dict(kernel=GROUP, split=False, rounds=False)),
    (3, 128, 1280, PAIR, dict(kernel=GROUP, split=False, rounds=False)),
    (5, 19072, 2048, m.Config(1, 0, 32), dict(kernel=FEW, split=True)),
    (64, 18944, 4096, PAIR, dict(kernel=FEW, split=True)),
]
GROUPS = [
    (3, [(9600, 1024)], dict(split=False, rounds=False)),
    (16, [(11008, 1024), (8192, 1536)], dict(split=False, rounds=True)),
    (20, [(4352, 1280)] * 5, dict(split=False, rounds=True)),
    (16, [(11008, 4096)] * 2, dict(split=True, rounds=True)),
    (5, [(4096, 4096), (11008, 4096), (4096, 11008)], dict(split=True, rounds=True)),
    (20, [(4352, 4352)] * 5, dict(split=True, rounds=True)),
    (7, [(11008, 3072), (8192, 3328)], dict(split=True, rounds=True)),
]


# dense inliers, one task per pair of CTAs -> form, do the outlier stages have a ring geometry of their own (slots: inliers', outliers')
KEEP7, DENSE2, ELEM = m.Config(1, m.gran_keep(7), 32), m.Config(2, m.GRAN_DENSE, 32), m.Config(1, m.GRAN_ELEM, 32)
RINGS = [
    (600, 5120, 6144, DENSE, FULL, (6, 8)),
    (600, 5120, 6400, KEEP7, FULL, (6, 8)),
    (2900, 1152, 6912, DENSE2, FULL, (6, 8)),
    (1100, 4096, 2304, KEEP7, TWO, (4, 6)),
    (1300, 3200, 2048, DENSE, TWO, (4, 6)),
    (4001, 1152, 3072, ELEM, TWO, (4, 6)),
    (1500, 4096, 11008, KEEP7, TWO, (4, 6)),
    # one-unit tasks with few stages, several tasks per pair, less than eight inlier stages, no outliers
    (600, 5120, 2048, DENSE, FULL, (6, 6)),
    (600, 5120, 2304, KEEP7, FULL, (6, 6)),
    (2900, 1152, 2816, DENSE2, FULL, (6, 6)),
    (387, 8192, 2048, ELEM, FULL, (6, 6)),
    (423, 6272, 3584, DENSE, FULL, (6, 6)),
    (4096, 4096, 16384, DENSE, FULL, (6, 6)),
    (2048, 2560, 1280, DENSE, TWO, (4, 4)),
    (600, 8192, 11008, m.Config(0, m.GRAN_DENSE, 32), TWO, (4, 4)),
]


def runs(plan, want):
    for name, value in want.items():
        got = plan.ksplit > 1 if name == "split" else getattr(plan, name)
        assert (bool(got) if isinstance(value, bool) else got) == value, name


@pytest.mark.parametrize("M,N,K,cfg,want", FORMS)
def test_shapes_take_the_forms_they_are_tested_for(M, N, K, cfg, want):
    runs(linear_plan(M, N, K, cfg, machine(*B200))[0], want)


@pytest.mark.parametrize("M,N,K,cfg,form,slots", RINGS)
def test_ring_geometries(M, N, K, cfg, form, slots):
    on = machine(*B200)
    r = linear_rings(M, N, K, cfg, on)
    runs(linear_plan(M, N, K, cfg, on)[0], dict(kernel=PAIRS, form=form))
    assert (r.slots, r.out_slots) == slots
    assert r.bytes == max(r.slots * r.slot_bytes, r.out_slots * r.out_slot_bytes) <= 227 * 1024
    assert (r.out_slot_bytes < r.slot_bytes) == (r.out_slots > r.slots)


@pytest.mark.parametrize("M,shapes,want", GROUPS)
def test_groups_are_dealt_out_as_tested(M, shapes, want):
    runs(group_plan(M, shapes, machine(*B200))[0], want)


def test_split_counts():
    """one, two and four thread blocks per left-over item, and two, three and four pairs per task, occur among the tested shapes"""
    on = machine(*B200)
    group = [linear_plan(*f[:4], on)[0] for f in FORMS if f[4]["kernel"] == GROUP] + [group_plan(M, sh, on)[0] for M, sh, _ in GROUPS]
    assert {1, 2, 4} == {p.ksplit for p in group} and {1, 2} <= {p.tail_items for p in group if p.ksplit > 1}
    assert {1, 3, 4} <= {linear_plan(*f[:4], on)[0].ksplit for f in FORMS if f[4]["kernel"] == PAIRS}


def test_plan_queries_refuse_what_the_calls_refuse():
    m.build()
    L, p, on = m.lib(), Plan(), machine(*B200)
    cfg, elem = m.Config(), m.Config(1, m.GRAN_ELEM, 64)
    ask = lambda M, N, K, c: L.sdq_diag_linear_plan(i64(M), i64(N), i64(K), ctypes.byref(c), 0, *on, ctypes.byref(p), None, i64(0))
    assert (ask(1, 128, 256, cfg), ask(0, 128, 256, cfg), ask(1, 100, 256, cfg), ask(1, 128, 200, cfg), ask(1, 128, 256, elem)) == (0, 2, 2, 2, 4)
    assert L.sdq_diag_group_plan(0, i64(1), None, None, *on, ctypes.byref(p), None, i64(0)) == 1


@pytest.mark.gpu
def test_the_device_at_hand_takes_the_same_forms():
    here = (ctypes.c_int(0), None)
    for M, N, K, cfg, want in FORMS:
        plan, tasks = linear_plan(M, N, K, cfg, here)
        runs(plan, want)
    for M, N, K, cfg, form, slots in RINGS:
        r = linear_rings(M, N, K, cfg, here)
        runs(linear_plan(M, N, K, cfg, here)[0], dict(kernel=PAIRS, form=form))
        assert (r.slots, r.out_slots) == slots
    for M, shapes, want in GROUPS:
        plan, segs = group_plan(M, shapes, here)
        runs(plan, want)
        cover_group(plan, segs, shapes)


def test_wide_tiles_are_split_over_two_pairs_at_most():
    """tiles of more tokens than an alternating accumulator has room for: K over one pair or two, in the form without alternation"""
    on, seen = machine(*B200), set()
    for M, N, K, cfg in [(500, 4096, 4096, PAIR), (470, 3840, 5120, PAIR), (512, 4096, 8192, UE), (500, 4096, 4096, DENSE), (500, 2048, 4096, PAIR), (8192, 1024, 1024, PAIR),
                         (500, 4096, 2048, PAIR), (256, 4096, 4096, PAIR), (1000, 2048, 4096, PAIR), (250, 8192, 4096, PAIR)]:
        plan, tasks = linear_plan(M, N, K, cfg, on)
        cover_pairs(plan, tasks, M, N)
        seen.add((plan.token_tile > 224, plan.ksplit))
        if plan.ksplit > 1 and plan.token_tile > 224:
            assert plan.ksplit == 2 and not plan.alternate and plan.tasks <= B200[1][0]
    assert (True, 2) in seen and (False, 1) in seen


@pytest.mark.parametrize("M,N,K,cfg,wide", [
    (240, 6528, 7680, m.Config(0, m.GRAN_DENSE, 32), False),
    (1068, 1408, 7424, m.Config(0, m.GRAN_DENSE, 32), False),
    (1259, 1024, 2560, KEEP7, False),
    (1711, 1024, 2816, DENSE, False),
    (1264, 1536, 3328, DENSE2, False),
    (211, 5376, 14336, m.Config(0, m.GRAN_DENSE, 32), True),
    (252, 7808, 7168, m.Config(0, m.GRAN_DENSE, 32), False),
    (236, 4864, 11520, m.Config(0, m.GRAN_DENSE, 32), False),
    (1118, 1280, 4608, ELEM, False),
    (450, 2944, 4608, DENSE, True),
    (919, 1920, 5888, DENSE, True),
    (211, 7424, 9216, ELEM, True),
    (1249, 1280, 3584, UE, True),
    (500, 4096, 4096, PAIR, True),
])
def test_which_wide_tiles_are_split(M, N, K, cfg, wide):
    """dense inliers: narrower tiles, with alternating accumulators, where these are the faster"""
    plan, _ = linear_plan(M, N, K, cfg, machine(*B200))
    assert (plan.ksplit == 2 and not plan.alternate) == wide
