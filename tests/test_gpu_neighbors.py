"""CUDA neighbour-table builder against the oracle: indices and distances bit-exact."""
import threading

import numpy as np
import pytest
import torch

import lantern_inputs as li
import oracle
import paper_2410_03355_b200 as lt

pytestmark = pytest.mark.gpu


def _gpu(cb, k):
    idx, dist = lt.build_neighbors(torch.from_numpy(cb).cuda(), k)
    torch.cuda.synchronize()
    return idx.cpu().numpy(), dist.cpu().numpy()


@pytest.mark.parametrize("V,D,k", [(1024, 8, 16), (1000, 8, 1), (520, 3, 520), (64, 1, 7), (2048, 8, 300),
                                   (777, 5, 100), (300, 32, 33)])
def test_small_d_exact(V, D, k):
    cb = li.codebook_gaussian(V, D, seed=21, normalise=(D > 1))
    gi, gd = _gpu(cb, k)
    oi, od = oracle.build_neighbors(cb, k)
    assert np.array_equal(gi, oi)
    assert np.array_equal(gd.view(np.uint32), od.view(np.uint32))


def test_ties_and_duplicates_exact():
    # integer codebook: massive exact ties, broken by index; duplicates of a code keep self first
    cb = li.codebook_integer(1500, 4, lo=-2, hi=3, seed=5)
    cb[700] = cb[3]
    for k in (2, 64, 999):
        gi, gd = _gpu(cb, k)
        oi, od = oracle.build_neighbors(cb, k)
        assert np.array_equal(gi, oi), k
        assert np.array_equal(gd, od), k
    const = np.ones((600, 8), np.float32)          # every distance is 0: order is pure index order
    gi, _ = _gpu(const, 50)
    oi, _ = oracle.build_neighbors(const, 50)
    assert np.array_equal(gi, oi)


def test_outliers_and_overflowing_distances_exact():
    # One code far away stretches the key range so that every other key falls into the select's first bin
    # (the crowded-bin path with all of its passes); codes of magnitude 1e30 make distances overflow to inf
    # (equal keys, ordered by index).
    cb = li.codebook_gaussian(3000, 8, seed=77)
    cb[1234] *= 1e15
    for k in (5, 300, 3000):
        gi, gd = _gpu(cb, k)
        oi, od = oracle.build_neighbors(cb, k)
        assert np.array_equal(gi, oi), k
        assert np.array_equal(gd.view(np.uint32), od.view(np.uint32)), k
    cb = li.codebook_gaussian(900, 4, seed=78)
    cb[::7] *= 1e30
    with np.errstate(over="ignore"):
        gi, gd = _gpu(cb, 200)
        oi, od = oracle.build_neighbors(cb, 200)
    assert np.array_equal(gi, oi)
    assert np.array_equal(gd.view(np.uint32), od.view(np.uint32))


@pytest.mark.parametrize("V,D,k", [(1100, 256, 64), (640, 40, 640), (2000, 100, 1000), (1001, 37, 100), (130, 33, 130)])
def test_large_d_exact(V, D, k):
    cb = li.codebook_clustered(V, D, centres=37, seed=8)
    gi, gd = _gpu(cb, k)
    oi, od = oracle.build_neighbors(cb, k)
    assert np.array_equal(gi, oi)
    assert np.array_equal(gd.view(np.uint32), od.view(np.uint32))


@pytest.mark.parametrize("name,k", [("batch_chain", 1000), ("single_image", 100), ("stress", 1000)])
def test_full_size_sampled_rows(name, k):
    # V = 16384 at the configurations' k: every row is built on the GPU, a seeded sample of
    # rows is recomputed by the oracle one by one; all rows are checked structurally.
    cb = li.config_codebook(name)
    V = cb.shape[0]
    gi, gd = _gpu(cb, k)
    rows = np.random.default_rng(3).choice(V, size=48, replace=False).astype(np.int32)
    oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi[rows], oi)
    assert np.array_equal(gd[rows].view(np.uint32), od.view(np.uint32))
    assert np.array_equal(gi[:, 0], np.arange(V))
    assert np.all(gd[:, 0] == 0) and np.all(np.diff(gd, axis=1) >= 0)
    assert gi.min() >= 0 and gi.max() < V
    srt = np.sort(gi, axis=1)
    assert np.all(srt[:, 1:] != srt[:, :-1])       # no token twice in a row


def test_argument_errors():
    cb = torch.from_numpy(li.codebook_gaussian(64, 8)).cuda()
    with pytest.raises(lt.LanternError) as e:
        lt.build_neighbors(cb, 65)
    assert e.value.code == -2
    with pytest.raises(lt.LanternError):
        lt.build_neighbors(cb, 0)
    with pytest.raises(ValueError):
        lt.build_neighbors(cb.cpu(), 4)


@pytest.mark.parametrize("V,D,k,kind", [
    (2048, 8, 1000, "gauss"), (2049, 8, 1000, "gauss"), (2049, 8, 1, "gauss"),      # the sampled bound starts at 2049 codes
    (4096, 8, 1000, "period"), (4096, 4, 300, "ties"),                              # codes of one cluster 512 apart; ties
    (6000, 8, 2500, "gauss"), (9001, 8, 4097, "gauss"),                             # four, two rows per CTA
    (2500, 40, 700, "period"), (5001, 33, 1500, "period"), (8193, 33, 4097, "gauss")])   # keys read from scratch
def test_selection_paths_exact(V, D, k, kind):
    if kind == "ties":
        cb = li.codebook_integer(V, D, lo=-2, hi=3, seed=9)
    elif kind == "period":
        cb = li.codebook_clustered(V, D, centres=512, seed=10)
    else:
        cb = li.codebook_gaussian(V, D, seed=11)
    gi, gd = _gpu(cb, k)
    rows = np.unique(np.concatenate([np.arange(20), np.arange(V - 20, V), np.random.default_rng(1).integers(0, V, 24)])).astype(np.int32)
    oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi[rows], oi)
    assert np.array_equal(gd[rows].view(np.uint32), od.view(np.uint32))
    assert np.array_equal(gi[:, 0], np.arange(V))
    srt = np.sort(gi, axis=1)
    assert np.all(srt[:, 1:] != srt[:, :-1])


@pytest.mark.parametrize("V,D,k,kind,with_dist", [
    (4096, 40, 1000, "period", True), (4099, 33, 100, "gauss", True), (4100, 36, 30, "gauss", False),   # every pair once, through lists
    (4096, 40, 300, "ties", True), (6144, 64, 700, "big clusters", True),                               # lists that fail
    (4096, 40, 1000, "period", False), (4095, 40, 100, "gauss", True)])                                 # no room for lists; too few codes
def test_lists_exact(V, D, k, kind, with_dist):
    if kind == "ties":
        cb = li.codebook_integer(V, D, lo=0, hi=2, seed=9)
    elif kind == "gauss":
        cb = li.codebook_gaussian(V, D, seed=11)
    else:
        cb = li.codebook_clustered(V, D, centres=512 if kind == "period" else 7, seed=10)
    idx, dist = lt.build_neighbors(torch.from_numpy(cb).cuda(), k, with_dist=with_dist)
    torch.cuda.synchronize()
    gi = idx.cpu().numpy()
    rows = np.unique(np.concatenate([np.arange(20), np.arange(V - 20, V), np.random.default_rng(1).integers(0, V, 24)])).astype(np.int32)
    oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi[rows], oi)
    if with_dist:
        assert np.array_equal(dist.cpu().numpy()[rows].view(np.uint32), od.view(np.uint32))
    assert np.array_equal(gi[:, 0], np.arange(V))
    srt = np.sort(gi, axis=1)
    assert np.all(srt[:, 1:] != srt[:, :-1])


# few codes: every key kept or a sampled bound, CTAs of two rows or of eight, lists or blocks of rows -- each line from both sides
@pytest.mark.parametrize("V,D,k", [
    (1024, 40, 500), (1025, 40, 500), (2304, 12, 2304), (2305, 12, 40), (2304, 13, 700), (2305, 13, 700), (3072, 8, 500), (3073, 8, 500),
    (2304, 64, 100), (2305, 64, 100), (2560, 45, 256), (2560, 45, 257), (4096, 33, 500), (4097, 33, 500)])
@pytest.mark.parametrize("kind", ["sphere", "ties", "nan"])
def test_few_codes_exact(V, D, k, kind):
    cb = li.codebook_integer(V, D, lo=0, hi=2, seed=3) if kind == "ties" else li.codebook_gaussian(V, D, seed=4)
    if kind == "nan":       # such a code is nobody's neighbour as long as there are others; which rows differ is not looked at
        cb[V // 2, 0] = np.nan
        if k == V:
            pytest.skip("every code is asked for")
    idx, dist = lt.build_neighbors(torch.from_numpy(cb).cuda(), k)
    torch.cuda.synchronize()
    rows = np.unique(np.concatenate([np.arange(9), np.arange(V - 9, V), np.random.default_rng(1).integers(0, V, 12)])).astype(np.int32)
    rows = rows[rows != V // 2]
    gi, gd = idx.cpu().numpy()[rows], dist.cpu().numpy()[rows]
    if kind == "nan":
        assert not np.any(gi == V // 2)
        other = np.delete(cb, V // 2, axis=0)
        oi, od = oracle.build_neighbors(other, k, rows=(rows - (rows > V // 2)).astype(np.int32))
        oi = oi + (oi >= V // 2)
    else:
        oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi, oi)
    assert np.array_equal(gd.view(np.uint32), od.view(np.uint32))


def test_host_threads_with_tables_of_different_size():
    """Tables whose rows need different amounts of shared memory, built by two host threads on streams of their own: the
    kernel's limit is common to both."""
    V, D, calls = 4000, 8, 3000
    cb = torch.from_numpy(li.codebook_gaussian(V, D, seed=12)).cuda()
    ks = (20, 700)
    want = [lt.build_neighbors(cb, k, with_dist=False)[0] for k in ks]
    got = [torch.empty_like(t) for t in want]
    torch.cuda.synchronize()
    lib = lt.load_library()
    codes = [None, None]

    def work(i, stream):
        torch.cuda.set_device(0)
        args = (cb.data_ptr(), V, D, ks[i], got[i].data_ptr(), None, None, 0, stream.cuda_stream)
        codes[i] = {lib.lantern_build_neighbors(*args) for _ in range(calls)}

    threads = [threading.Thread(target=work, args=(i, torch.cuda.Stream())) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert codes == [{0}, {0}]
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("V,D,k,with_dist", [
    (2400, 8, 200, True), (9000, 8, 1000, True), (4500, 16, 2500, False),      # keys computed: CTAs of two rows, of eight, of four
    (2600, 40, 300, False), (6000, 33, 1500, False),                          # read from scratch
    (4096, 40, 500, True), (4400, 36, 30, True)])                             # every pair once, through lists
@pytest.mark.parametrize("dead", ["first", "last", "mixed", "all", "few values"])
def test_many_equal_codes_exact(V, D, k, with_dist, dead):
    """Codes that are the same (dead ones): more keys equal a row's bound than it takes, and those of the smallest index count."""
    rng = np.random.default_rng(V + k)
    cb = rng.standard_normal((V, D)).astype(np.float32)
    if dead == "few values":
        cb = cb[rng.integers(0, 5, V)]
    else:
        at = {"first": np.arange(V // 2), "last": np.arange(V // 2, V), "mixed": rng.permutation(V)[:V // 2], "all": np.arange(V)}[dead]
        cb[at] = cb[0]
    cb = np.ascontiguousarray(cb)
    idx, dist = lt.build_neighbors(torch.from_numpy(cb).cuda(), k, with_dist=with_dist)
    torch.cuda.synchronize()
    gi = idx.cpu().numpy()
    rows = np.unique(np.concatenate([np.arange(12), np.arange(V // 2 - 6, V // 2 + 6), np.arange(V - 12, V), rng.integers(0, V, 24)])).astype(np.int32)
    oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi[rows], oi)
    if with_dist:
        assert np.array_equal(dist.cpu().numpy()[rows].view(np.uint32), od.view(np.uint32))
    assert np.array_equal(gi[:, 0], np.arange(V))
    srt = np.sort(gi, axis=1)
    assert np.all(srt[:, 1:] != srt[:, :-1])


@pytest.mark.parametrize("V,D,k,kind", [
    (8192, 8, 300, "gauss"), (8191, 16, 300, "period"), (6145, 13, 64, "gauss"), (6144, 16, 64, "gauss"), (8193, 32, 200, "gauss"),
    (16384, 4, 30, "ties"), (12289, 20, 1000, "period")])
def test_steps_of_the_key_pass_exact(V, D, k, kind):
    """Four codes per thread and step where the number of steps of two is even, two elsewhere: on either side, full and ragged."""
    if kind == "ties":
        cb = li.codebook_integer(V, D, lo=-2, hi=3, seed=9)
    elif kind == "period":
        cb = li.codebook_clustered(V, D, centres=512, seed=10)
    else:
        cb = li.codebook_gaussian(V, D, seed=11)
    gi, gd = _gpu(cb, k)
    rows = np.unique(np.concatenate([np.arange(12), np.arange(V - 12, V), np.random.default_rng(1).integers(0, V, 24)])).astype(np.int32)
    oi, od = oracle.build_neighbors(cb, k, rows=rows)
    assert np.array_equal(gi[rows], oi)
    assert np.array_equal(gd[rows].view(np.uint32), od.view(np.uint32))
