"""Calls at the edges of a rule that once answered them slowly or unsafely:
one test per rule."""
from __future__ import annotations

import itertools
import math
import time

import numpy as np
import pytest

from tests.helpers import F32_RTOL, random_data

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


# more combinations at or above a threshold than the collecting pass has room
# for (2^20): it ends at an item that all its warps know, without waiting for
# loads that nothing takes (a wait of two seconds a stage), and every score is
# looked at instead
@pytest.mark.parametrize("k,n,m", [(2, 1600, 200), (3, 200, 300), (4, 80, 130), (5, 50, 260)])
@pytest.mark.parametrize("variant", ["auto", "separate"])
def test_threshold_found_too_often(epi, ctx, k, n, m, variant):
    ds = epi.Dataset(ctx, *random_data(n, m, seed=n))

    def timed(chunk):
        t = time.perf_counter()
        r, found = epi.search_threshold(ds, k, 1e-9, 100, chunk=chunk, with_counts=False)
        return r, found, time.perf_counter() - t

    ctx.set_tc_variant(variant)
    try:
        want, n_want, t_want = timed(math.comb(n, k))
        assert n_want > 1 << 20
        for _ in range(2):
            got, n_got, t_got = timed(0)
            assert n_got == n_want
            assert (got.rank == want.rank).all() and (got.mi == want.mi).all()
            assert t_got < t_want + 1.5
    finally:
        ctx.set_tc_variant("auto")
        ds.close()


# a pipeline wait that runs out ends the search with an error at every order
# and variant, whichever role's wait it was, and the context stays usable (a
# wait may also be met within the first look at its barrier, whatever the limit)
@pytest.mark.parametrize("k,n,m", [(2, 300, 3000), (3, 90, 3000), (4, 60, 3000), (5, 23, 3000)])
@pytest.mark.parametrize("variant", ["auto", "separate"])
def test_wait_limit_at_every_order(epi, k, n, m, variant):
    own = epi.Context(0)
    own.set_tc_variant(variant)
    ds = epi.Dataset(own, *random_data(n, m, seed=n))
    want = epi.search(ds, k, 20, path="popc")
    for limit in (1, 0):
        own.set_wait_limit(limit)
        try:
            got = epi.search(ds, k, 20, path="tc")
            assert (got.rank == want.rank).all() and (got.mi == want.mi).all()
        except epi.EpiError as e:
            assert limit == 1 and e.status == epi.EPI_ETIMEOUT
    ds.close()
    own.close()


# studies with pair tiles are searched by themselves, except where eight or more
# of a batch save little by them: a replayed graph launches nothing that the
# context counts, a search of its own does
@pytest.mark.parametrize("k,n,m,count,alone", [(4, 45, 1000, 8, 0), (4, 45, 1000, 7, 7), (4, 60, 900, 9, 0),
                                               (4, 45, 4000, 8, 8), (4, 100, 1000, 8, 8), (5, 26, 300, 8, 8)])
def test_batch_searches_studies_alone(epi, k, n, m, count, alone):
    own = epi.Context(0)
    sets = [epi.Dataset(own, *random_data(n, m, seed=n + i)) for i in range(count)]
    sets.append(epi.Dataset(own, *random_data(30, 200, seed=1)))
    orders = [k] * count + [3]
    want = [epi.search(s, o, 20, path="popc") for s, o in zip(sets, orders)]
    epi.search_batched(own, sets, orders, [20] * len(sets))
    before = own.kernel_launches()
    epi.search(sets[0], k, 20, path="tc")
    each = own.kernel_launches() - before
    before = own.kernel_launches()
    got = epi.search_batched(own, sets, orders, [20] * len(sets))
    assert own.kernel_launches() - before == alone * each
    for a, b in zip(got, want):
        assert (a.rank == b.rank).all() and (a.mi == b.mi).all() and (a.counts == b.counts).all()
    own.close()


# the work space of a large search with pair tiles (5.4 GiB here) is given back
# behind it; a small one stays with the context
def test_pair_space_is_given_back(epi):
    import torch
    own = epi.Context(0)
    small = epi.Dataset(own, *random_data(60, 300, seed=1))
    large = epi.Dataset(own, *random_data(160, 300, seed=2))
    want = epi.search(large, 3, 10, path="tc")          # the operand and the scratch are there
    epi.search(small, 5, 10)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    a = epi.search(large, 5, 10)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 1 << 30
    b = epi.search(large, 5, 10)
    assert (a.rank == b.rank).all() and (a.mi == b.mi).all()
    assert (epi.search(large, 3, 10, path="tc").rank == want.rank).all()
    own.close()


# a search that finds no room for pair tiles runs without them
def test_no_room_for_pair_space(epi):
    own = epi.Context(0)
    ds = epi.Dataset(own, *random_data(60, 300, seed=1))
    want = epi.search(ds, 4, 10, path="popc")
    epi.search(ds, 3, 10, path="tc")
    epi.search(ds, 4, 10, path="tc", rank_range=(0, 480000))   # the operand and the scratch are there
    own.inject_alloc_failure(0)
    got = epi.search(ds, 4, 10, path="tc")
    own.inject_alloc_failure(-1)
    assert (got.rank == want.rank).all() and (got.mi == want.mi).all()
    own.close()


# a search captured into a graph, of a study that was never searched: order 2
# chooses the tensor path from 100 SNPs, whose operand a capture cannot build
def test_captured_search_of_a_new_study(epi):
    import torch
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        own = epi.Context(0)
        warm, ds = (epi.Dataset(own, *random_data(200, 400, seed=i)) for i in (1, 2))
        out = torch.zeros(10 * epi.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        n_out = torch.zeros(1, dtype=torch.int32, device="cuda")
        status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        # the context's scratch is there
        epi.search_async(warm, 2, 10, out, None, n_out, status, path="popc")
        epi.search_async(warm, 2, 10, out, None, n_out, status)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            epi.search_async(ds, 2, 10, out, None, n_out, status)
        want = epi.search(ds, 2, 10)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = np.frombuffer(out.cpu().numpy().tobytes(), dtype=epi.RESULT_DTYPE)
        assert int(status.item()) == 0 and int(n_out.item()) == 10
        assert (got["rank"] == want.rank).all() and (got["mi"] == want.mi).all()
        del graph
        own.close()


# a search that a stream capture refuses (the tensor path's operand is not
# there) leaves the study and the context as they were
def test_search_after_a_refused_capture(epi):
    import torch
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        own = epi.Context(0)
        warm, ds = (epi.Dataset(own, *random_data(120, 400, seed=i)) for i in (1, 2))
        want = epi.search(ds, 3, 10, path="popc")
        out = torch.zeros(10 * epi.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        n_out = torch.zeros(1, dtype=torch.int32, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        epi.search_async(warm, 3, 10, out, None, n_out, status)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        with pytest.raises(epi.EpiError):
            epi.search_async(ds, 3, 10, out, None, n_out, status, path="tc")
        with pytest.raises(RuntimeError):
            graph.capture_end()
        for _ in range(2):
            got = epi.search(ds, 3, 10, path="tc")
            assert (got.rank == want.rank).all() and (got.mi == want.mi).all() and (got.counts == want.counts).all()
        del graph
        own.close()


# the autotuner times the tensor path as searches run it, with pair tiles where
# they apply (from 40 SNPs at order 4): its two passes then launch as many
# kernels more than those of a study without them as two searches do
def test_autotuner_times_pair_tiles(epi):
    counts = []
    for n in (39, 40):
        own = epi.Context(0)
        ds = epi.Dataset(own, *random_data(n, 300, seed=n))
        epi.search(ds, 4, 10, path="tc")
        start = own.kernel_launches()
        epi.autotune(ds, 4)
        tuned = own.kernel_launches()
        epi.search(ds, 4, 10, path="tc")
        counts.append((tuned - start, own.kernel_launches() - tuned))
        own.close()
    (tune39, search39), (tune40, search40) = counts
    assert search40 > search39
    assert tune40 - tune39 == 2 * (search40 - search39)


# at orders 7-8 the autotuner's shapes are those of kernels that neither
# searches nor batches take: it must not spend more on them than on a few
# searches (a few shapes, two passes each)
@pytest.mark.parametrize("k,n,m,times", [(7, 20, 1000, 17), (8, 20, 1000, 40)])
def test_autotuner_at_high_orders(epi, k, n, m, times):
    own = epi.Context(0)
    ds = epi.Dataset(own, *random_data(n, m, seed=k))

    def seconds(f):
        f()
        t = time.perf_counter()
        f()
        return time.perf_counter() - t

    search = seconds(lambda: epi.search(ds, k, 100))
    assert seconds(lambda: epi.autotune(ds, k)) < times * search
    own.close()


# a pass that writes every score launches its kernel alone: nothing selects the
# best of the scores
@pytest.mark.parametrize("k,n,m", [(1, 50, 300), (2, 40, 300), (5, 12, 200), (6, 12, 200)])
def test_every_score_alone(epi, ctx, k, n, m):
    ds = epi.Dataset(ctx, *random_data(n, m, seed=k))
    before = ctx.kernel_launches()
    scores = epi.score_all(ds, k).cpu().numpy()
    assert ctx.kernel_launches() - before == (2 if k >= 6 else 1)
    best = epi.search(ds, k, 10, path="popc")
    assert (scores[best.rank.astype(np.int64)] == best.mi_f32).all()
    ds.close()


# the last level of a merge sorts up to 512 entries by counting, more by a
# bitonic sort: both sides, equal scores, and pools cut down by the selection
@pytest.mark.parametrize("k", [1, 2, 511, 512, 513, 1000, 1025, 4096])
@pytest.mark.parametrize("levels", [3, 100000])
def test_sorted_topk(epi, ctx, k, levels):
    import torch
    rng = np.random.default_rng(k + levels)
    x = (rng.integers(0, levels, 20000) / 16.0 - 1.0).astype(np.float32)
    s, i = epi.topk(ctx, torch.from_numpy(x).cuda(), k)
    want = np.lexsort((np.arange(len(x)), -x))[:k]
    assert (np.asarray(i.cpu()).astype(np.int64) == want).all()
    assert (s.cpu().numpy() == x[want]).all()


@pytest.mark.parametrize("top_n", [400, 500, 700, 1024])
def test_merge_of_large_pools(epi, ctx, top_n):
    ds = epi.Dataset(ctx, *random_data(90, 300, seed=top_n))
    a, b = epi.search(ds, 3, top_n, path="tc"), epi.search(ds, 3, top_n, path="popc")
    assert len(a) == top_n and (a.rank == b.rank).all() and (a.mi == b.mi).all()
    ds.close()


def _copies(n, cases, copies, seed):
    """Controls that repeat the cases: every score is zero."""
    half, _ = random_data(n, cases, seed=seed)
    geno = np.concatenate([half] * (1 + copies), axis=1)
    return geno, (np.arange(geno.shape[1]) < cases).astype(np.uint8)


# scores too small for the table of n ln n: all of SNPs with one genotype (zero
# without a count), a few others (a list, without such SNPs), more cells in all
# than those of 1024 tables and one in 64 (the popcount path)
@pytest.mark.parametrize("k,n,kind", [(3, 60, "constant"), (4, 30, "constant"), (3, 40, "half"), (4, 22, "half"),
                                      (3, 40, "balanced"), (4, 22, "balanced"), (4, 40, "balanced"),
                                      (3, 19, "copies"), (3, 20, "copies"), (3, 60, "copies"), (4, 25, "copies")])
def test_small_scores(epi, ctx, k, n, kind):
    if kind == "copies":
        geno, pheno = _copies(n, 70, 2, n)
    elif kind == "balanced":
        # two SNPs whose carriers are shared out evenly among constant ones and others
        geno, pheno = random_data(n, 300, seed=n, m1=150)
        geno[::2] = 1
        cases, ctrls = np.nonzero(pheno == 1)[0], np.nonzero(pheno == 0)[0]
        geno[0, cases[:1]] = geno[0, ctrls[:1]] = 2
        geno[2, cases[5:8]] = geno[2, ctrls[9:12]] = 0
    else:
        geno, pheno = random_data(n, 300, seed=n)
        geno[::2 if kind == "half" else 1] = np.arange(len(geno[::2 if kind == "half" else 1]))[:, None] % 3
    ds = epi.Dataset(ctx, geno, pheno)
    got = epi.score_all(ds, k).cpu().numpy().astype(np.float64)
    combs = np.array(list(itertools.combinations(range(n), k)), dtype=np.uint32)
    _, want = epi.score_tables(ds, k, epi.tables(ds, combs))
    assert (np.abs(got - want) <= F32_RTOL * want + 1e-9 * (want > 0)).all()
    assert (got[want == 0] == 0).all()
    assert kind in ("half", "balanced") or (want == 0).all()
    ds.close()


# a table of nothing but such scores costs no more than a few of the popcount
# path's (which finds the best of them by ranges of the ranks)
@pytest.mark.parametrize("k,n,m", [(3, 250, 300), (4, 80, 300)])
@pytest.mark.parametrize("kind", ["constant", "copies"])
def test_small_scores_are_quick(epi, ctx, k, n, m, kind):
    def seconds(ds, f):
        f()
        best = 1e9
        for _ in range(3):
            t = time.perf_counter()
            f()
            best = min(best, time.perf_counter() - t)
        ds.close()
        return best

    plain = epi.Dataset(ctx, *random_data(n, m, seed=1))
    usual = seconds(plain, lambda: epi.search_threshold(plain, k, 1e9, 1, chunk=math.comb(n, k)))
    if kind == "copies":
        geno, pheno = _copies(n, m // 3, 2, 1)
    else:
        geno, pheno = np.zeros((n, m), np.uint8), (np.arange(m) % 2).astype(np.uint8)
    ds = epi.Dataset(ctx, geno, pheno)
    assert seconds(ds, lambda: epi.score_all(ds, k)) < 2 * usual


# rare variants put most individuals into one cell of an order-6 table: the
# search must not take much longer than on common ones
def test_high_order_rare_variants(epi, ctx):
    times = []
    for p in ((0.05, 0.5), (0.001, 0.01)):
        ds = epi.Dataset(ctx, *random_data(36, 2048, seed=3, m1=1024, p_levels=p))
        best = 1e9
        for _ in range(3):
            t = time.perf_counter()
            epi.search(ds, 6, 20)
            best = min(best, time.perf_counter() - t)
        times.append(best)
        ds.close()
    assert times[1] < 1.3 * times[0]
