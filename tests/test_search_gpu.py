"""GPU parity of the batched beam search (Sec. 2.1, Algorithm 1) against the
CPU oracle, through the C ABI.

uint8 data: ids, int32 distances, evaluation and expansion counts bit-exact.
fp32 data: >= 99.9% of (query, rank) ids equal, distances within 1e-5
relative (1e-5 of |x||q| for inner product), recall@10 within 0.001."""
import json
import math
import os

import numpy as np
import pytest

import oracle
from paper_2506_15986_gb300 import ann, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import make_index, search  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2506_15986_gb300 import _build
    _build.build()
    ann.load_library()


@pytest.fixture(scope="module")
def c1():
    w = synth.small_u8()
    g, _ = oracle.build_graph(w["base"], K=64, R=32, alpha=1.0)
    med = oracle.medoid(w["base"])
    h = make_index(w["base"], g, med)
    yield dict(w, graph=g, medoid=med, h=h)
    ann.ann_free_index(h)


def _oracle(w, q, L, k, **kw):
    return oracle.search(w["base"], w["graph"], np.asarray(q, np.float64),
                         kw.pop("entries", w["medoid"]), L, k, **kw)


def test_toy_graphs_exact(golden_dir):
    with open(os.path.join(golden_dir, "toy_graphs.json")) as f:
        cases = json.load(f)["cases"]
    for c in cases:
        pts = np.asarray(c["points"], np.float32)
        pad = np.zeros((len(pts), 4), np.float32)
        pad[:, : pts.shape[1]] = pts  # zero padding keeps squared L2 unchanged
        q = np.zeros((1, 4), np.float32)
        q[0, : pts.shape[1]] = c["query"]
        h = make_index(pad, np.asarray(c["adjacency"], np.int32), c["entry"])
        try:
            ids, d, ev, hp, st = search(h, q, c["k"], c["L"], W=c["W"])
        finally:
            ann.ann_free_index(h)
        assert st == ann.OK
        assert ids[0].tolist() == c["ids"], c["name"]
        exp = [math.inf if v == "inf" else float(v) for v in c["dists"]]
        assert d[0].tolist() == exp, c["name"]
        assert (int(ev[0]), int(hp[0])) == (c["evals"], c["hops"]), c["name"]


@pytest.mark.parametrize("L,W", [(64, 1), (16, 1), (128, 1), (64, 2), (512, 2), (10, 1),
                                 (64, 3), (128, 4), (512, 4), (1024, 4), (2048, 2), (4096, 2)])
def test_c1_u8_bit_exact(c1, L, W):
    q = c1["queries"]
    k = min(10, L)
    ids, d, ev, hp, st = search(c1["h"], q, k, L, W=W)
    oi, od, oe, oh = _oracle(c1, q, L, k, W=W)
    assert st == ann.OK
    assert np.array_equal(ids, oi)
    assert np.array_equal(d, od.astype(np.int64).clip(max=2**31 - 1).astype(np.int32))
    assert np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("R,W", [(100, 1), (64, 2), (128, 1)])
def test_u8_wide_rows_bit_exact(c1, R, W):
    # unpruned K-NN graphs with up to 128 neighbour slots per step: ragged
    # last slot (R = 100), and steps whose survivors need the 128-key sort
    base = c1["base"][:4000]
    g, _ = oracle.knn(base, base.astype(np.float64), R, exclude=np.arange(len(base), dtype=np.int32))
    med = oracle.medoid(base)
    h = make_index(base, g, med)
    try:
        q = c1["queries"]
        ids, d, ev, hp, st = search(h, q, 10, 96, W=W)
    finally:
        ann.ann_free_index(h)
    oi, od, oe, oh = oracle.search(base, g, q.astype(np.float64), med, 96, 10, W=W)
    assert st == ann.OK
    assert np.array_equal(ids, oi)
    assert np.array_equal(d, od.astype(np.int64).astype(np.int32))
    assert np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("team,stage_rows,gather", [(1, 32, 1), (2, 4, 1), (4, 8, 1), (16, 16, 1), (32, 5, 1),
                                                    (4, 8, 4), (8, 5, 4), (2, 12, 4), (32, 16, 4), (4, 1, 4)])
def test_c1_team_sizes_bit_exact(c1, team, stage_rows, gather):
    # every distance team size, gather round size and fetch mode (a bulk copy
    # per row, or TMA tensor gathers of four rows with ragged rounds padded)
    # gives the same exact int32 distances, hence the same search
    q = c1["queries"]
    ids, d, ev, hp, st = search(c1["h"], q, 10, 128, W=2, team=team, stage_rows=stage_rows, gather=gather)
    oi, od, oe, oh = _oracle(c1, q, 128, 10, W=2)
    assert st == ann.OK
    assert np.array_equal(ids, oi) and np.array_equal(ev, oe) and np.array_equal(hp, oh)
    assert np.array_equal(d, od.astype(np.int64).astype(np.int32))


def test_forced_wait_timeout_is_reported_and_recoverable(c1):
    # fault injection: every wait for gathered rows gives up at once.  Each
    # query fails with -1 ids, the call reports a timeout, the copies in
    # flight still land, and the next normal call on the same index is exact.
    q = c1["queries"]
    ids, d, ev, hp, st = search(c1["h"], q, 10, 64, flags=ann.SEARCH_FAULT_WAIT)
    assert st == ann.ERR_TIMEOUT
    assert (ids == -1).all() and (d == 2**31 - 1).all()
    ids, d, ev, hp, st = search(c1["h"], q, 10, 64)
    oi, od, oe, oh = _oracle(c1, q, 64, 10)
    assert st == ann.OK
    assert np.array_equal(ids, oi) and np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("L,spill_bits,hash_bits", [(128, 0, 8), (512, 10, 8), (128, 0, -1), (512, 10, -1)])
def test_c1_spill_to_global_table_stays_exact(c1, L, spill_bits, hash_bits):
    # hash_bits=8: 192 shared slots, far fewer than the evaluations, so the
    # exact global spill table carries most of the visited set; with
    # spill_bits=10 at L=512 most queries pass 768 evaluations and move on to
    # the second, 4x larger table
    q = c1["queries"]
    ids, d, ev, hp, st = search(c1["h"], q, 10, L, hash_bits=hash_bits, spill_bits=spill_bits)
    oi, od, oe, oh = _oracle(c1, q, L, 10)
    assert st == ann.OK
    assert (oe > 192).mean() > 0.8  # most queries outgrow the shared table
    if spill_bits:
        assert (oe > 768).mean() > 0.5  # ... and the first global one
    assert np.array_equal(ids, oi) and np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("spill_bits", [10, 12])
def test_visited_tables_kept_in_l2_change_nothing(c1, spill_bits):
    # ANN_SEARCH_VISITED_L2 only changes where the first-level visited tables
    # live in the cache: the search stays bit-exact
    q = c1["queries"]
    ids, d, ev, hp, st = search(c1["h"], q, 10, 96, W=2, hash_bits=-1, spill_bits=spill_bits,
                                flags=ann.SEARCH_VISITED_L2)
    oi, od, oe, oh = _oracle(c1, q, 96, 10, W=2)
    assert st == ann.OK
    assert np.array_equal(ids, oi) and np.array_equal(ev, oe) and np.array_equal(hp, oh)
    assert np.array_equal(d, od.astype(np.int64).astype(np.int32))


@pytest.mark.parametrize("nq,m,n_hubs", [(20_000, 1, 8), (6_000, 4, 1_500), (1, 1, 1), (5_000, 1, 5_000)])
def test_grouped_work_order_changes_nothing(c1, nq, m, n_hubs):
    # ANN_SEARCH_GROUP_ENTRIES only changes the order in which the teams take
    # the work items (sorted by a hash of the first seed): every item's ids,
    # distances and counters stay bit-exact at its own index.  Batches larger
    # than the sort's 4,096 buckets and 1,024 threads, few and many distinct
    # first seeds, seed sets, per-query k and L.
    rng = np.random.default_rng(nq + m)
    q = np.tile(c1["queries"], (nq // len(c1["queries"]) + 1, 1))[:nq]
    hubs = rng.choice(len(c1["base"]), n_hubs, replace=False)
    seeds = hubs[rng.integers(0, n_hubs, (nq, m))].astype(np.int32)
    if m > 1:
        seeds[:, 1:][rng.random((nq, m - 1)) < 0.3] = -1
    Ls = rng.integers(10, 97, nq).astype(np.int32)
    ks = np.minimum(rng.integers(1, 11, nq), Ls).astype(np.int32)
    ent = seeds if m > 1 else seeds[:, 0]
    ids, d, ev, hp, st = search(c1["h"], q, 10, 96, W=2, entries=ent, ks=ks, Ls=Ls,
                                flags=ann.SEARCH_GROUP_ENTRIES)
    oi, od, oe, oh = oracle.search(c1["base"], c1["graph"], q.astype(np.float64), ent, 0, 0, W=2,
                                   Ls=Ls, ks=ks)
    assert st == ann.OK
    oi_full = np.full((nq, 10), -1, np.int32)
    oi_full[:, : oi.shape[1]] = oi
    assert np.array_equal(ids, oi_full)
    assert np.array_equal(ev, oe) and np.array_equal(hp, oh)
    od_full = np.zeros((nq, 10), np.int64)
    od_full[:, : od.shape[1]] = np.where(np.isfinite(od), od, 0).astype(np.int64)
    valid = oi_full >= 0
    assert np.array_equal(d[valid], od_full[valid].astype(np.int32))


def test_grouped_work_order_with_a_bad_seed(c1):
    # a seed out of range fails its own item only, wherever the sort put it
    q = np.tile(c1["queries"], (30, 1))
    seeds = np.full(len(q), c1["medoid"], np.int32)
    seeds[1234] = len(c1["base"])
    ids, d, ev, hp, st = search(c1["h"], q, 10, 64, entries=seeds, flags=ann.SEARCH_GROUP_ENTRIES)
    assert st == ann.ERR_INVALID_ARG
    assert (ids[1234] == -1).all()
    ok = np.arange(len(q)) != 1234
    oi, od, oe, oh = _oracle(c1, q[ok], 64, 10)
    assert np.array_equal(ids[ok], oi) and np.array_equal(ev[ok], oe)


def test_c1_per_query_entries_k_L(c1):
    rng = np.random.default_rng(3)
    q = c1["queries"]
    nq = len(q)
    entries = rng.integers(0, len(c1["base"]), nq).astype(np.int32)
    Ls = rng.integers(10, 200, nq).astype(np.int32)
    ks = np.minimum(rng.integers(1, 11, nq), Ls).astype(np.int32)
    ids, d, ev, hp, st = search(c1["h"], q, 10, 200, entries=entries, ks=ks, Ls=Ls)
    oi, od, oe, oh = oracle.search(c1["base"], c1["graph"], q.astype(np.float64), entries, 0, 0,
                                   Ls=Ls, ks=ks)
    assert st == ann.OK
    oi_full = np.full((nq, 10), -1, np.int32)
    oi_full[:, : oi.shape[1]] = oi
    assert np.array_equal(ids, oi_full)
    assert np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("m,W", [(2, 1), (4, 4), (32, 2)])
def test_c1_seed_sets_bit_exact(c1, m, W):
    # seed sets with unused slots (-1) and repeated seeds: the initial pool
    # holds every distinct seed, evaluated once
    rng = np.random.default_rng(m)
    q = c1["queries"]
    seeds = rng.integers(0, len(c1["base"]), (len(q), m)).astype(np.int32)
    seeds[rng.random(seeds.shape) < 0.3] = -1
    seeds[:, 0] = np.where(seeds[:, 0] < 0, c1["medoid"], seeds[:, 0])
    if m > 1:
        seeds[::3, 1] = seeds[::3, 0]  # a repeated seed
    ids, d, ev, hp, st = search(c1["h"], q, 10, 64, W=W, entries=seeds)
    oi, od, oe, oh = oracle.search(c1["base"], c1["graph"], q.astype(np.float64), seeds, 64, 10, W=W)
    assert st == ann.OK
    assert np.array_equal(ids, oi) and np.array_equal(ev, oe) and np.array_equal(hp, oh)
    assert np.array_equal(d, od.astype(np.int64).astype(np.int32))


def test_c1_label_mode_targets(c1):
    q = c1["queries"][:50]
    t, _ = oracle.knn(c1["base"], q.astype(np.float64), 1)
    rng = np.random.default_rng(5)
    entries = rng.integers(0, len(c1["base"]), 50).astype(np.int32)
    entries[0] = t[0, 0]  # entry is the target: 1 evaluation, 0 expansions
    ids, d, ev, hp, st = search(c1["h"], q, 1, 64, entries=entries, targets=t[:, 0])
    _, _, oe, oh = oracle.search(c1["base"], c1["graph"], q.astype(np.float64), entries, 64, 1,
                                 targets=t[:, 0])
    assert st == ann.OK
    assert np.array_equal(ev, oe) and np.array_equal(hp, oh)
    assert (ev[0], hp[0]) == (1, 0)


def test_empty_batch_and_bad_device_inputs(c1):
    q = c1["queries"]
    ids, d, ev, hp, st = search(c1["h"], q[:0], 10, 64)
    assert ids.shape == (0, 10) and st == ann.OK
    # a per-query L above the launch maximum is reported, never read past
    ids, d, ev, hp, st = search(c1["h"], q[:4], 10, 64, Ls=np.array([64, 65, 64, 64]))
    assert st == ann.ERR_INVALID_ARG
    assert (ids[1] == -1).all() and (ids[0] >= 0).all()
    assert ann.ann_sync_status(c1["h"]) == ann.OK  # cleared by the read
    # host-side parameter checks return before any launch
    for kw in (dict(team=3), dict(team=64), dict(stage_rows=33), dict(W=5), dict(hash_bits=7), dict(hash_bits=-2),
               dict(spill_bits=9), dict(spill_bits=17), dict(flags=16), dict(gather=2),
               dict(entries=np.zeros((4, 33), np.int32))):
        with pytest.raises(ann.AnnError) as e:
            search(c1["h"], q[:4], 10, 64, **kw)
        assert e.value.status == ann.ERR_INVALID_ARG, kw
    # a seed row without any node, or with an id out of range, fails on the device
    for bad in ([-1, -1], [5, len(c1["base"])]):
        ids, d, ev, hp, st = search(c1["h"], q[:1], 10, 64, entries=np.array([bad], np.int32))
        assert st == ann.ERR_INVALID_ARG and (ids == -1).all()


@pytest.fixture(scope="module")
def f32_case():
    w = synth.shift_f32(n=20000, nq=300, n_train=0)
    g, _ = oracle.build_graph(w["base"], K=64, R=32)
    med = oracle.medoid(w["base"])
    h = make_index(w["base"], g, med)
    yield dict(w, graph=g, medoid=med, h=h)
    ann.ann_free_index(h)


def _f32_parity(ids, d, oi, od, truth, scale=None):
    agree = (ids == oi).mean()
    assert agree >= 0.999, agree
    ok = ids == oi
    ref = np.abs(od) if scale is None else scale[:, None].repeat(od.shape[1], 1)
    rel = np.abs(d.astype(np.float64) - od)[ok] / np.maximum(ref[ok], 1e-30)
    assert rel.max() <= 1e-5, rel.max()
    r_gpu = oracle.recall_at_k(ids, truth, 10)
    r_or = oracle.recall_at_k(oi, truth, 10)
    assert abs(r_gpu - r_or) <= 1e-3


@pytest.mark.parametrize("L,W,team,gather", [(32, 1, 0, 0), (64, 1, 0, 0), (128, 2, 0, 0), (128, 2, 2, 0),
                                            (128, 4, 32, 0), (96, 4, 4, 4), (128, 4, 8, 4)])
def test_f32_l2_parity(f32_case, L, W, team, gather):
    q = f32_case["queries"]
    ids, d, ev, hp, st = search(f32_case["h"], q, 10, L, W=W, team=team, gather=gather)
    oi, od, oe, oh = _oracle(f32_case, q, L, 10, W=W)
    truth, _ = oracle.knn(f32_case["base"], q.astype(np.float64), 10)
    assert st == ann.OK
    _f32_parity(ids, d, oi, od, truth)
    assert (ev == oe).mean() >= 0.99 and (hp == oh).mean() >= 0.99


def test_f32_ip_parity():
    w = synth.ip_f32(n=12000, nq=200)
    base = w["base"]
    # graph built on L2 over unit vectors (same order as IP for unit norms)
    g, _ = oracle.build_graph(base, K=48, R=32)
    med = oracle.medoid(base)
    h = make_index(base, g, med, metric=ann.IP)
    try:
        q = w["queries"]
        ids, d, ev, hp, st = search(h, q, 10, 64)
    finally:
        ann.ann_free_index(h)
    oi, od, oe, oh = oracle.search(base, g, q.astype(np.float64), med, 64, 10, metric=oracle.IP)
    truth, _ = oracle.knn(base, q.astype(np.float64), 10, metric=oracle.IP)
    scale = np.linalg.norm(q.astype(np.float64), axis=1)  # |x| = 1
    assert st == ann.OK
    _f32_parity(ids, d, oi, od, truth, scale=scale)


def test_visited_set_outgrows_both_global_tables():
    # points on a line, x_i = i, each node linked to the next 64: a search
    # from node 0 walks the chain and evaluates every node up to a little past
    # the query.  At L = 16 the shared table (1,024 slots) and the first
    # global table (4,096) overflow; the 4x larger one takes up to 12,288
    # keys, so the query at 6,000 still finishes exactly and the one at
    # 14,000 (all 14,000 nodes) fails with a capacity status and -1 ids.
    n, R = 14000, 64
    base = np.zeros((n, 4), np.float32)
    base[:, 0] = np.arange(n)
    nb = np.arange(n)[:, None] + 1 + np.arange(R)[None, :]
    g = np.where(nb < n, nb, -1).astype(np.int32)
    q = np.zeros((3, 4), np.float32)
    q[:, 0] = [2000, 6000, 14000]
    h = make_index(base, g, 0)
    try:
        ids, d, ev, hp, st = search(h, q, 10, 16, hash_bits=10)
    finally:
        ann.ann_free_index(h)
    assert st == ann.ERR_CAPACITY
    oi, od, oe, oh = oracle.search(base, g, q[:2].astype(np.float64), 0, 16, 10)
    assert oe[1] > 3 * 4096 // 4  # past the first global table
    assert np.array_equal(ids[:2], oi) and np.array_equal(ev[:2], oe) and np.array_equal(hp[:2], oh)
    assert np.array_equal(d[:2], od.astype(np.float32))
    assert (ids[2] == -1).all()


@pytest.mark.parametrize("nq", [1, 153, 1_217, 4_865])
@pytest.mark.parametrize("L,W", [(20, 4), (160, 2), (2_000, 4)])
def test_default_sizes_change_nothing(c1, nq, L, W):
    # the visited table and gather rounds chosen when the caller leaves them
    # open depend on nq and L (all queries resident, SMs part full, SMs full);
    # results never do
    q = np.resize(c1["queries"], (nq, 128))
    oi, od, oe, oh = _oracle(c1, c1["queries"][:min(nq, 100)], L, 10, W=W)
    ids, d, ev, hp, st = search(c1["h"], q, 10, L, W=W)
    assert st == ann.OK
    at = np.arange(nq) % 100
    assert np.array_equal(ids, oi[at]) and np.array_equal(ev, oe[at]) and np.array_equal(hp, oh[at])
    assert np.array_equal(d, od[at].astype(np.int64).astype(np.int32))


@pytest.mark.parametrize("hash_bits", [0, -1, 8])
def test_tables_sized_by_each_querys_own_L(hash_bits):
    # on a random graph nearly every neighbour is new, so a query outgrows the
    # table its own L sizes (3,072 keys up to L = 76) and moves to the second
    # one, whose size is the launch's
    rng = np.random.default_rng(12)
    w = synth.small_u8(n=20_000)
    g = rng.integers(0, 20_000, size=(20_000, 32)).astype(np.int32)
    q = w["queries"]
    Ls = np.resize(np.array([1, 40, 76, 77, 300, 512], np.int32), len(q))
    ks = np.minimum(Ls, 10).astype(np.int32)
    h = make_index(w["base"], g, 0)
    try:
        ids, d, ev, hp, st = search(h, q, 10, 512, W=4, ks=ks, Ls=Ls, hash_bits=hash_bits)
    finally:
        ann.ann_free_index(h)
    oi, od, oe, oh = oracle.search(w["base"], g, q.astype(np.float64), 0, 512, 10, W=4, Ls=Ls, ks=ks)
    assert st == ann.OK
    assert (oe[Ls == 76] > 3_072).any()
    assert np.array_equal(ids, oi[:, :10]) and np.array_equal(ev, oe) and np.array_equal(hp, oh)


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("metric", [ann.L2, ann.IP])
@pytest.mark.parametrize("dim,team", [(72, 0), (104, 0), (128, 0), (136, 0), (200, 0), (256, 0), (256, 8), (128, 4), (256, 32), (8, 0), (64, 0), (68, 0)])
def test_distance_forms_are_bit_identical(dtype, metric, dim, team):
    # rows read one by one are summed by fewer lanes than the team has, or
    # several rows at once, by the row's chunks and the type; tensor gathers
    # always take a row at a time by the whole team: the same bits either way, for
    # every step width and the last, ragged round
    rng = np.random.default_rng(dim + team)
    n = 3_000
    if dtype == np.float16:
        dim *= 2
    base = rng.standard_normal((n, dim)).astype(dtype)
    q = rng.standard_normal((150, dim)).astype(np.float32)
    g = rng.integers(0, n, size=(n, 29)).astype(np.int32)
    h = make_index(base, g, 5, metric=metric)
    try:
        for W in (1, 2, 4):
            a = search(h, q, 20, 40, W=W, team=team, gather=1)
            for gather in (0, 4):  # left open: tensor gathers up to 256 bytes a row
                b = search(h, q, 20, 40, W=W, team=team, gather=gather)
                assert a[4] == b[4] == ann.OK
                for x, y in zip(a[:4], b[:4]):
                    assert np.array_equal(x.view(np.int32), y.view(np.int32))
    finally:
        ann.ann_free_index(h)


@pytest.mark.parametrize("metric", [ann.L2, ann.IP])
@pytest.mark.parametrize("dim", [496, 1_000, 1_008])
def test_int8_distance_forms_are_bit_identical(metric, dim):
    # as above for int8 rows with their scale (teams of 8 and 16); rows of 1,000
    # codes end in zero codes
    rng = np.random.default_rng(dim)
    n = 2_000
    x = torch.from_numpy(rng.standard_normal((n, dim)).astype(np.float32)).cuda()
    packed = torch.empty((n, ann.ann_i8s_row_bytes(dim)), dtype=torch.uint8, device="cuda:0")
    q = rng.standard_normal((150, dim)).astype(np.float32)
    g = rng.integers(0, n, size=(n, 29)).astype(np.int32)
    ann.ann_quantize_i8s(x, n, dim, packed)
    h = ann.ann_index_create(packed, g, 5, ann.I8S, metric, n=n, dim=dim, degree=29)
    try:
        for W in (1, 4):
            a = search(h, q, 20, 40, W=W, gather=1)
            b = search(h, q, 20, 40, W=W, gather=4)
            assert a[4] == b[4] == ann.OK
            for u, v in zip(a[:4], b[:4]):
                assert np.array_equal(u.view(np.int32), v.view(np.int32))
    finally:
        ann.ann_free_index(h)


def test_small_spill_tables_of_a_large_batch():
    # about 4,800 evaluations a query: more than the global tables of spill_bits =
    # 10 hold, so the shared table stays although it costs the batch occupancy
    rng = np.random.default_rng(1)
    x = rng.standard_normal((5_000, 16)).astype(np.float32)
    g = rng.integers(0, 5_000, size=(5_000, 32)).astype(np.int32)
    q = rng.standard_normal((5_000, 16)).astype(np.float32)
    h = make_index(x, g, 0)
    try:
        a = search(h, q, 10, 512, W=4)
        b = search(h, q, 10, 512, W=4, spill_bits=10)
    finally:
        ann.ann_free_index(h)
    assert a[4] == ann.OK and b[4] == ann.OK
    assert a[2].max() > 3072 and all(np.array_equal(u, v) for u, v in zip(a[:4], b[:4]))


def test_searches_of_two_threads(f32_case):
    # one index, searched by two threads with small and with large pools (whose
    # shared memory differs): every search launches, with its usual results
    import threading
    q = f32_case["queries"][:100]
    out = {}

    def run(L):
        h, dq, s = f32_case["h"], torch.from_numpy(q).to("cuda:0"), torch.cuda.Stream()
        ids = torch.empty((100, 10), dtype=torch.int32, device="cuda:0")
        dd = torch.empty((100, 10), device="cuda:0")
        p = ann.search_params(10, L, W=4)
        torch.cuda.synchronize()
        try:
            for _ in range(3000):
                ann.ann_search_batch(h, dq, 100, None, p, ids, dd, stream=s)
                s.synchronize()
            out[L] = ids.cpu().numpy()
        except ann.AnnError as e:
            out[L] = e
    threads = [threading.Thread(target=run, args=(L,)) for L in (16, 1024)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for L in (16, 1024):
        assert not isinstance(out[L], ann.AnnError), out[L]
        assert np.array_equal(out[L], search(f32_case["h"], q, 10, L, W=4)[0])


def _long_rows(dtype, dim, nq):
    """An index of 960-d rows and a function that times a search of it (ms)."""
    rng = np.random.default_rng(dim)
    x = rng.standard_normal((5_000, dim)).astype(np.float32)
    g = rng.integers(0, 5_000, size=(5_000, 32)).astype(np.int32)
    dx = torch.from_numpy(x).to("cuda:0")
    rows = dx.half()
    if dtype == ann.I8S:
        rows = torch.empty((5_000, ann.ann_i8s_row_bytes(dim)), dtype=torch.uint8, device="cuda:0")
        ann.ann_quantize_i8s(dx, 5_000, dim, rows)
    h = ann.ann_index_create(rows, torch.from_numpy(g).to("cuda:0"), 0, dtype, n=5_000, dim=dim, degree=32)
    q = dx.repeat(2, 1)[:nq].contiguous()
    ids = torch.empty((nq, 10), dtype=torch.int32, device="cuda:0")
    dd = torch.empty((nq, 10), device="cuda:0")

    def ms(**knobs):
        p = ann.search_params(10, 16, W=4, **knobs)
        out = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ann.ann_search_batch(h, q, nq, None, p, ids, dd)
            b.record()
            b.synchronize()
            out.append(a.elapsed_time(b))
        return min(out[2:]), ids.clone()
    return h, ms


@pytest.mark.parametrize("dtype,team", [(ann.F16, 2), (ann.I8S, 4)])
def test_open_rounds_fill_the_warp(dtype, team):
    # a small team fixed, the round left open: as many rows as the warp takes at
    # once, so no slower than asking for rounds of sixteen
    h, ms = _long_rows(dtype, 960, 6_000)
    try:
        (a, ia), (b, ib) = ms(team=team, hash_bits=-1), ms(team=team, hash_bits=-1, stage_rows=16)
        assert torch.equal(ia, ib) and a <= 1.1 * b, (a, b)
        ms(team=1)  # 32 rows at once: the longest round, or what fits
    finally:
        ann.ann_free_index(h)


def test_short_rounds_keep_every_team_busy():
    # rounds of as many rows as the warp has teams: a row each, not two for half of
    # them (rounds of four took 1.27 times what rounds of eight take here)
    h, ms = _long_rows(ann.I8S, 960, 1)
    try:
        (a, ia), (b, ib) = ms(team=8, stage_rows=4), ms(team=8, stage_rows=8)
        assert torch.equal(ia, ib) and a <= 1.27 * b, (a, b)
    finally:
        ann.ann_free_index(h)


@pytest.mark.parametrize("R,L,W,knobs,mixed", [(32, 512, 4, dict(hash_bits=13, spill_bits=12), False),
                                               (32, 512, 2, dict(hash_bits=11, spill_bits=10), False),
                                               (128, 282, 1, {}, True), (128, 282, 1, dict(hash_bits=13), True)])
def test_visited_keys_survive_a_smaller_first_table(R, L, W, knobs, mixed):
    # a shared table that outgrows the first global one: asked for so, or by a query
    # whose own L is small; no node is evaluated twice, as with tables that are
    # never left
    rng = np.random.default_rng(R)
    n = 12_000
    x = rng.standard_normal((n, 16)).astype(np.float32)
    g = rng.integers(0, n, size=(n, R)).astype(np.int32)
    q = rng.standard_normal((200, 16)).astype(np.float32)
    own = dict(Ls=rng.integers(10, L + 1, size=200), ks=np.full(200, 10)) if mixed else {}
    h = make_index(x, g, 0)
    try:
        a = search(h, q, 10, L, W=W, hash_bits=-1, spill_bits=16, **own)
        b = search(h, q, 10, L, W=W, **knobs, **own)
    finally:
        ann.ann_free_index(h)
    small = own["Ls"] <= 76 if mixed else slice(None)
    assert a[4] == ann.OK and a[2][small].max() > (1536 if knobs.get("hash_bits") == 11 else 6144)
    if knobs.get("spill_bits") == 10:  # 3,072 keys at most: failed queries say so
        assert b[4] in (ann.OK, ann.ERR_CAPACITY)
        done = b[0][:, 0] >= 0
    else:
        assert b[4] == ann.OK
        done = np.ones(200, bool)
    assert all(np.array_equal(u[done], v[done]) for u, v in zip(a[:4], b[:4]))
