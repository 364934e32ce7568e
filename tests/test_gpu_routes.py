"""Calls that reach a kernel or a branch by a rule on their sizes, on both
sides of the rule: the tensor path's pair tiles, its class shift, order 2's
automatic path, thresholds and whole score tables counted on the tensor
cores, merges of small and large pools, batches with studies searched alone,
and the fused training kernels."""
from __future__ import annotations

import itertools
import math

import numpy as np
import pytest

from oracle import mlp as M
from oracle import oracle as O
from tests.helpers import F32_RTOL, check_topn, random_data
from tests.test_gpu_learn import _bf16, _grad_magnitudes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def epi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_02460_gb300 import epi as E
    E.load()
    return E


@pytest.fixture(scope="module")
def ctx(epi):
    return epi.Context(0)


def _same(a, b):
    """Two routes of one search: the same records, bit for bit."""
    assert (a.rank == b.rank).all() and (a.combs == b.combs).all()
    assert (a.mi == b.mi).all() and (a.counts == b.counts).all()


# pair tiles start at 40 SNPs (order 4) and 24 (order 5); one SNP fewer takes
# the other tiles.  Odd SNP and sample counts, one class small, both variants.
@pytest.mark.parametrize("k,n,m,m1,variant", [
    (4, 39, 300, 130, "auto"), (4, 40, 300, 130, "auto"), (4, 41, 257, 20, "auto"), (4, 42, 300, 130, "separate"),
    (4, 75, 513, 256, "auto"), (5, 23, 270, 140, "auto"), (5, 24, 270, 140, "auto"), (5, 25, 129, 11, "separate"),
    (5, 27, 1000, 900, "auto")])
def test_pair_tiles(epi, ctx, k, n, m, m1, variant):
    geno, pheno = random_data(n, m, seed=100 * k + n, m1=m1)
    ds = epi.Dataset(ctx, geno, pheno)
    ctx.set_tc_variant(variant)
    try:
        if math.comb(n, k) * 2 * 3 ** k * 4 < 1 << 30:
            got = epi.debug_counts(ds, k)
            combs = np.array(list(itertools.combinations(range(n), k)), dtype=np.uint32)
            for i in range(0, len(combs), 50000):
                assert (got[i:i + 50000] == epi.tables(ds, combs[i:i + 50000])).all()
        _same(epi.search(ds, k, 50, path="tc"), epi.search(ds, k, 50, path="popc"))
    finally:
        ctx.set_tc_variant("auto")


# the classes share an accumulator while c1 2^p + c0 < 2^24 with 2^p > c0 + 1
# (c1, c0: the largest counts of a genotype): 4094 each is the last equal pair
@pytest.mark.parametrize("m1,m0", [(4094, 4094), (4095, 4095), (4094, 4095), (3, 8190), (8190, 3)])
@pytest.mark.parametrize("k,n", [(2, 12), (3, 12), (4, 40)])
def test_class_shift_limit(epi, ctx, k, n, m1, m0):
    geno, pheno = random_data(n, m1 + m0, seed=m1 + n, m1=m1)
    geno[:4] = 0          # one cell of the first combinations holds everyone
    ds = epi.Dataset(ctx, geno, pheno)
    first = np.arange(k, dtype=np.uint32)[None]
    assert epi.tables(ds, first)[0, :, 0].tolist() == O.tables(geno, pheno, first.astype(np.int32))[0, :, 0].tolist()
    _same(epi.search(ds, k, 40, path="tc"), epi.search(ds, k, 40, path="popc"))
    if k < 4:
        combs = np.array(list(itertools.combinations(range(n), k)), dtype=np.uint32)
        assert (epi.debug_counts(ds, k) == epi.tables(ds, combs)).all()


# the automatic path of order 2 changes at 100 SNPs
@pytest.mark.parametrize("n,m,m1", [(99, 333, None), (100, 333, None), (121, 64, 5), (241, 130, 125)])
def test_order2_automatic_path(epi, ctx, n, m, m1):
    geno, pheno = random_data(n, m, seed=n, m1=m1)
    ds = epi.Dataset(ctx, geno, pheno)
    r = epi.search(ds, 2, 64)
    _same(r, epi.search(ds, 2, 64, path="popc"))
    oc, om, _ = O.search(geno, pheno, 2, 64)
    check_topn(r.combs, r.mi, oc, om)


# merges: one entry, fewer combinations than asked for (990) and a few more (1035)
@pytest.mark.parametrize("k,n,top_n", [(2, 120, 1), (2, 130, 2), (2, 45, 1024), (2, 46, 1024), (3, 40, 1000)])
def test_merge_sizes(epi, ctx, k, n, top_n):
    geno, pheno = random_data(n, 200, seed=top_n)
    ds = epi.Dataset(ctx, geno, pheno)
    a, b = epi.search(ds, k, top_n, path="tc"), epi.search(ds, k, top_n, path="popc")
    assert len(a) == min(top_n, math.comb(n, k))
    _same(a, b)


# chunk 0 screens on the tensor cores, a chunk size takes every score
@pytest.mark.parametrize("k,n,m,m1", [(2, 50, 200, None), (3, 33, 700, None), (3, 30, 129, 9), (4, 22, 300, 150),
                                      (5, 15, 90, 50)])
def test_threshold_routes(epi, ctx, k, n, m, m1):
    geno, pheno = random_data(n, m, seed=k * n, m1=m1)
    ds = epi.Dataset(ctx, geno, pheno)
    best = epi.search(ds, k, 40)
    # in the widest gap among the best scores; above the best there is nothing;
    # below zero everything qualifies
    cut = 1 + int(np.argmax(best.mi[:-1] - best.mi[1:]))
    for thr, want in ((0.5 * float(best.mi[cut - 1] + best.mi[cut]), cut), (float(best.mi[0]) * 1.01, 0), (-1.0, math.comb(n, k))):
        a, na = epi.search_threshold(ds, k, thr, 60)
        b, nb = epi.search_threshold(ds, k, thr, 60, chunk=1000)
        assert (na, nb) == (want, want) and len(a) == min(60, na)
        _same(a, b)


# whole tables of orders 3-4: counted on the tensor cores and scored in fixed
# point, within the FP32 path's bound of the 64-bit score
@pytest.mark.parametrize("k,n,m,m1", [(3, 3, 50, None), (3, 41, 257, 30), (3, 25, 2999, 1500), (4, 4, 64, 32),
                                      (4, 23, 129, 100), (3, 20, 3500, 1700)])
def test_whole_score_tables(epi, ctx, k, n, m, m1):
    geno, pheno = random_data(n, m, seed=n + m, m1=m1)
    geno[1] = 2           # a SNP with one genotype: empty cells
    ds = epi.Dataset(ctx, geno, pheno)
    got = epi.score_all(ds, k).cpu().numpy().astype(np.float64)
    combs = np.array(list(itertools.combinations(range(n), k)), dtype=np.int32)
    want = np.array([O.mi(x[0], x[1], m) for x in O.tables(geno, pheno, combs)])
    assert (np.abs(got - want) <= F32_RTOL * np.abs(want) + 1e-9).all(), np.abs(got - want).max()


# a study large enough for pair tiles is searched by itself within a batch
@pytest.mark.parametrize("n_alone", [1, 2])
def test_batch_with_studies_alone(epi, ctx, n_alone):
    shapes = [(3, 30, 200), (2, 60, 150)] + [(4, 40 + i, 260) for i in range(n_alone)] + [(4, 20, 100)]
    dss = [epi.Dataset(ctx, *random_data(n, m, seed=n)) for _, n, m in shapes]
    orders = [k for k, _, _ in shapes]
    for _ in range(2):
        got = epi.search_batched(ctx, dss, orders, [20] * len(dss))
        for r, ds, k in zip(got, dss, orders):
            _same(r, epi.search(ds, k, 20, path="popc"))


# without room for the tensor path's operand the automatic choice answers by
# the popcount path
@pytest.mark.parametrize("call", ["search", "threshold", "scores"])
def test_no_room_for_the_operand(epi, call):
    geno, pheno = random_data(110, 200, seed=5)
    k = 2 if call == "search" else 3
    want_ctx, ctx = epi.Context(0), epi.Context(0)

    def run(c, ds):
        if call == "search":
            return epi.search(ds, k, 30)
        if call == "threshold":
            return epi.search_threshold(ds, k, 0.06, 100)[0]
        return epi.score_all(ds, k).cpu().numpy()

    a = run(want_ctx, epi.Dataset(want_ctx, geno, pheno))
    ds = epi.Dataset(ctx, geno, pheno)
    run(ctx, epi.Dataset(ctx, geno, pheno))   # the context's scratch is there
    ctx.inject_alloc_failure(0)
    b = run(ctx, ds)
    ctx.inject_alloc_failure(-1)
    if call == "scores":
        np.testing.assert_allclose(a, b, rtol=2 * F32_RTOL, atol=2e-9)
    else:
        _same(a, b)


# fused training kernels: rows around a tile and beyond one tile a block
# (512 x 32), inputs and hidden units at the rule's edges; (33 inputs, 288
# hidden units: the separate kernels).  Bounds as for the gradients of other
# shapes: differing terms of BF16 storage, FP32 sums, masks near zero.
@pytest.mark.parametrize("rows,n_in,hidden", [(1, 1, 32), (31, 5, 32), (33, 32, 96), (100, 33, 64), (65, 30, 288),
                                              (257, 30, 256), (16417, 7, 64)])
def test_fused_gradients(epi, ctx, rows, n_in, hidden):
    import torch
    rng = np.random.default_rng(rows)
    net = epi.MLP(ctx, n_in, hidden, seed=rows)
    theta = net.params().astype(np.float64)
    X = rng.standard_normal((rows, n_in)).astype(np.float32)
    y, (_, _, _, _, H2, _, W3) = M.forward(theta, X, n_in, hidden, rnd=_bf16)
    scale = np.abs(H2) @ np.abs(W3) + 1.0
    t = (y + 4.0 * scale * np.where(np.arange(rows) % 2 == 0, 1.0, -1.0)).astype(np.float32)
    g, loss = net.gradients(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda())
    g2, loss2 = net.gradients(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda())
    assert (g == g2).all()
    want = M.gradients(theta, X, t, n_in, hidden, rnd=_bf16, rnd_dz=_bf16)
    S, L, A = _grad_magnitudes(theta, X, t, n_in, hidden, _bf16)
    err = np.abs(g.astype(np.float64) - want)
    assert (err <= 2.0 ** -6 * L + 2.0 ** -12 * S + A + 1e-30).all()
    assert abs(loss - M.loss(theta, X, t, n_in, hidden, rnd=_bf16)) <= 1e-4 * abs(loss) + 1e-7
    net.close()


# the autotuner's choice moves a study between the batch's launches and a
# search of its own: the same batch before and after
def test_batch_after_new_choices(epi, tmp_path):
    own = epi.Context(0)
    sets = [epi.Dataset(own, *random_data(n, 300, seed=n)) for n in (60, 20, 50)]
    orders = [4, 3, 4]
    want = [epi.search(s, k, 20, path="popc") for s, k in zip(sets, orders)]
    epi.autotune(sets[0], 4)
    file = str(tmp_path / "tune.txt")
    epi.tune_save(own, file)
    with open(file) as f:
        lines = [x.split() for x in f.read().splitlines() if x and x[0] != "#"]
    for path in (2, 1, 2):
        with open(file, "w") as f:
            f.writelines(" ".join(x[:4] + [str(path)] + x[5:]) + "\n" for x in lines)
        epi.tune_load(own, file)
        for _ in range(2):
            for a, b in zip(epi.search_batched(own, sets, orders, [20] * 3), want):
                _same(a, b)
    own.close()


# orders 6-8 by histogram: items past a class's words, one individual in a
# class, eight and sixteen items a thread, counts past the logarithms kept in
# shared memory (1024), everyone in one cell, more samples than it takes
@pytest.mark.parametrize("k,n,m,m1", [
    (6, 9, 31, 1), (6, 13, 300, 299), (7, 10, 64, 32), (8, 10, 33, 16), (8, 9, 4096, 2048), (7, 10, 4097, 2100),
    (7, 9, 5000, 4990), (6, 9, 6000, 3000), (8, 9, 16384, 8000), (7, 9, 16500, 8000)])
@pytest.mark.parametrize("rare", [False, True])
def test_high_orders_by_histogram(epi, ctx, k, n, m, m1, rare):
    geno, pheno = random_data(n, m, seed=k + m, m1=m1, p_levels=(0.001, 0.02) if rare else (0.2, 0.5))
    geno[0] = 1
    ds = epi.Dataset(ctx, geno, pheno)
    combs = np.array(list(itertools.combinations(range(n), k)), dtype=np.int32)
    tables = O.tables(geno, pheno, combs)
    want = np.array([O.mi(x[0], x[1], m) for x in tables])
    assert (epi.tables(ds, combs.astype(np.uint32)) == tables).all()
    got = epi.score_all(ds, k).cpu().numpy().astype(np.float64)
    assert (np.abs(got - want) <= F32_RTOL * want + 1e-12).all(), np.abs(got - want).max()
    total = len(combs)
    for r0, r1 in ((0, total), (total // 3, total - 1)):
        r = epi.search(ds, k, 8, path="popc", rank_range=(r0, r1))
        oc, om, _ = O.search(geno, pheno, k, 8, rank_begin=r0, rank_end=r1)
        check_topn(r.combs, r.mi, oc, om)
        assert (r.counts == tables[r.rank.astype(np.int64)]).all()
        assert (np.abs(r.mi_f32 - want[r.rank.astype(np.int64)]) <= F32_RTOL * r.mi + 1e-12).all()


# controls that repeat the cases' genotypes `copies` times: every score is
# zero, and rank order decides (for these sizes the fixed-point logarithms
# leave a positive remainder)
@pytest.mark.parametrize("k,n,cases,copies", [(6, 16, 70, 2), (7, 16, 70, 2), (8, 16, 42, 4)])
def test_high_orders_without_association(epi, ctx, k, n, cases, copies):
    half, _ = random_data(n, cases, seed=k)
    geno = np.concatenate([half] * (1 + copies), axis=1)
    pheno = (np.arange(geno.shape[1]) < cases).astype(np.uint8)
    ds = epi.Dataset(ctx, geno, pheno)
    r = epi.search(ds, k, 10, path="popc")
    assert (r.mi == 0).all() and (r.mi_f32 == 0).all()
    assert (r.rank == np.arange(10)).all()
    assert float(epi.score_all(ds, k).abs().max()) == 0.0
    ds.close()


# the same at orders 3 and 4 (every score from the table of n ln n, which
# leaves up to 19 of its units here), and one SNP whose classes differ by one
# individual: scores far below the table's accuracy
@pytest.mark.parametrize("k", [3, 4])
@pytest.mark.parametrize("cases,copies", [(70, 2), (42, 4), (101, 1)])
def test_score_tables_without_association(epi, ctx, k, cases, copies):
    half, _ = random_data(9, cases, seed=k)
    geno = np.concatenate([half] * (1 + copies), axis=1)
    pheno = (np.arange(geno.shape[1]) < cases).astype(np.uint8)
    ds = epi.Dataset(ctx, geno, pheno)
    assert float(epi.score_all(ds, k).abs().max()) == 0.0
    geno = np.zeros((9, 2990), np.uint8)
    geno[3, :700] = 1
    geno[3, 1495:2194] = 1
    ds.close()
    ds = epi.Dataset(ctx, geno, (np.arange(2990) < 1495).astype(np.uint8))
    got = epi.score_all(ds, k).cpu().numpy()
    want = np.array([epi.search(ds, k, 1, path="popc", rank_range=(r, r + 1)).mi[0] for r in range(math.comb(9, k))])
    assert (want > 0).sum() == math.comb(8, k - 1)
    assert (np.abs(got - want) <= F32_RTOL * want).all()
    ds.close()


# one SNP with a single individual's difference between the classes, the
# others constant: scores far below 2^-19 keep their relative accuracy
@pytest.mark.parametrize("k,m", [(6, 3000), (7, 8000), (8, 8000), (8, 16000)])
def test_high_orders_smallest_scores(epi, ctx, k, m):
    geno = np.zeros((k + 1, m), np.uint8)
    geno[3, :m // 4 + 1] = 1
    geno[3, m // 2:m // 2 + m // 4] = 1
    pheno = (np.arange(m) < m // 2).astype(np.uint8)
    ds = epi.Dataset(ctx, geno, pheno)
    r = epi.search(ds, k, k + 1, path="popc")
    assert (r.mi[:k] > 0).all() and r.mi[k] == 0
    assert (np.abs(r.mi_f32 - r.mi) <= F32_RTOL * r.mi).all()
    ds.close()
