"""dt_batch: many independent clouds in one sequence of launches, every cloud bit-exact against the
oracle run on that cloud alone (the perturbed Delaunay triangulation is unique, so batching,
block shape and round size cannot change it)."""
import time

import numpy as np
import pytest

import oracle
from paper_1805_08831_gb300 import synth
from tests.inputs import DEGENERATE_SETS

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1805_08831_gb300 as dt  # noqa: E402


def run_batch(clouds, seed=0):
    off = np.zeros(len(clouds) + 1, dtype=np.uint64)
    off[1:] = np.cumsum([len(c) for c in clouds])
    xyz = np.ascontiguousarray(np.concatenate(clouds, axis=0), dtype=np.float64)
    with dt.Triangulation(seed=seed) as t:
        t.batch(torch.from_numpy(xyz).cuda(), off)
        tets, coff = t.tets_batch(canonical=True)
        st = t.stats()
    return [tets[int(coff[c]):int(coff[c + 1])] for c in range(len(clouds))], st


def split(xyz, off):
    return [xyz[int(off[c]):int(off[c + 1])] for c in range(len(off) - 1)]


def assert_clouds_match(clouds, got):
    for c, x in enumerate(clouds):
        ref, _ = oracle.delaunay(x)
        if not np.array_equal(got[c], ref):
            raise AssertionError(f"cloud {c} ({len(x)} points): {len(got[c])} vs {len(ref)} tetrahedra")


def test_batch_of_uneven_uniform_clouds_matches_oracle():
    xyz, off = synth.batched_clouds(48, 11, lo=50, hi=6000)
    clouds = split(xyz, off)
    got, st = run_batch(clouds)
    assert_clouds_match(clouds, got)
    assert st["n_clouds_degenerate"] == 0
    assert st["batch_warps"] in (4, 8, 16, 32)
    assert st["n_unique"] == len(xyz)


def test_batch_clouds_spanning_several_brio_rounds():
    # 2048 / 14336 / 100352 are the first BRIO round ends: these clouds use three rounds
    clouds = [synth.uniform_cube(n, 300 + n) for n in (2047, 2049, 14337, 30000)]
    got, _ = run_batch(clouds, seed=5)
    assert_clouds_match(clouds, got)


def test_batch_of_degenerate_clouds_and_duplicates():
    clouds = [DEGENERATE_SETS[k] for k in sorted(DEGENERATE_SETS)]
    mix = synth.degenerate_mix(6000, 7)
    mix[-500:] = mix[:500]  # duplicates inside the cloud
    clouds.append(mix)
    clouds.append(synth.cube_and_slab(5000, 9))
    got, st = run_batch(clouds)
    assert_clouds_match(clouds, got)
    assert st["n_exact"] > 0 and st["n_sos"] > 0


def test_batch_cloud_without_volume_is_skipped_not_fatal():
    plane = np.c_[synth.uniform_cube(200, 1)[:, :2], np.zeros(200)]
    clouds = [synth.uniform_cube(300, 2), plane, synth.uniform_cube(4, 3), synth.uniform_cube(5, 4)]
    got, st = run_batch(clouds)
    assert st["n_clouds_degenerate"] == 1
    assert len(got[1]) == 0
    for c in (0, 2, 3):
        ref, _ = oracle.delaunay(clouds[c])
        assert np.array_equal(got[c], ref)


def test_batch_equals_single_cloud_inserts():
    xyz, off = synth.batched_clouds(6, 21, lo=500, hi=20000)
    clouds = split(xyz, off)
    got, _ = run_batch(clouds, seed=3)
    for c, x in enumerate(clouds):
        with dt.Triangulation(seed=3) as t:
            t.insert(torch.from_numpy(np.ascontiguousarray(x)).cuda())
            single = t.tets_numpy()
        assert np.array_equal(got[c], single)


def test_batch_output_into_page_locked_host_memory():
    """Unsorted rows written by the collection kernel straight into page-locked host memory hold
    each cloud's tetrahedra (the sorted device output, as sets); pageable memory is refused by
    the C ABI and the binding falls back to its own array."""
    xyz, off = synth.batched_clouds(12, 41, lo=50, hi=6000)
    with dt.Triangulation(seed=3) as t:
        t.batch(torch.from_numpy(xyz).cuda(), off)
        ref, roff = t.tets_batch(canonical=True)
        pinned = torch.zeros((len(ref) + 7, 4), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
        got, goff = t.tets_batch(canonical=False, out=pinned)
        assert np.shares_memory(got, pinned) and np.array_equal(goff, roff)
        assert not pinned[len(ref):].any()
        pageable, poff = t.tets_batch(canonical=False, out=np.zeros((len(ref), 4), dtype=np.uint32))
        assert np.array_equal(poff, roff)
    for res in (got, pageable):
        for c in range(len(roff) - 1):
            a = np.sort(res[int(roff[c]):int(roff[c + 1])], axis=1)
            b = np.sort(ref[int(roff[c]):int(roff[c + 1])], axis=1)
            assert np.array_equal(a[np.lexsort(a.T[::-1])], b[np.lexsort(b.T[::-1])])


@pytest.mark.parametrize("warps", [8, 16, 32])
def test_every_block_shape_gives_the_same_tets(warps, monkeypatch):
    monkeypatch.setenv("DT_BATCH_WARPS", str(warps))
    monkeypatch.setenv("DT_BATCH_ALPHA", "0.3")
    xyz, off = synth.batched_clouds(20, 31, lo=50, hi=4000)
    clouds = split(xyz, off)
    got, st = run_batch(clouds)
    assert st["batch_warps"] == warps
    assert_clouds_match(clouds, got)


def test_batch_at_scale_sampled_clouds():
    """4096 clouds, sizes log-uniform in [50, 50000]: every cloud's tetrahedron count and a
    sample of clouds checked element by element against the oracle."""
    xyz, off = synth.batched_clouds(4096, 4)
    with dt.Triangulation(seed=0) as t:
        t.batch(torch.from_numpy(xyz).cuda(), off)
        tets, coff = t.tets_batch(canonical=True)
        st = t.stats()
    assert st["n_clouds_degenerate"] == 0 and st["device_error"] == 0
    assert st["n_unique"] == len(xyz)
    # between n and 7 n tetrahedra per cloud (about 6.7 n for large uniform clouds)
    counts = np.diff(coff.astype(np.int64))
    sizes = np.diff(off.astype(np.int64))
    assert np.all(counts > sizes) and np.all(counts < 7 * sizes)
    rng = np.random.default_rng(0)
    for c in rng.choice(4096, 12, replace=False):
        x = xyz[int(off[c]):int(off[c + 1])]
        ref, _ = oracle.delaunay(x)
        assert np.array_equal(tets[int(coff[c]):int(coff[c + 1])], ref), c


def test_repeated_batch_replays_its_graph_on_new_data():
    """The second call with the same buffer and cloud sizes replays the captured CUDA graph; the
    graph computes everything that depends on the coordinates on the device, so new values in
    the same buffer give their own triangulations."""
    xyz, off = synth.batched_clouds(30, 41, lo=50, hi=3000)
    xd = torch.from_numpy(xyz).cuda()
    with dt.Triangulation(seed=0) as t:
        t.batch(xd, off)
        first, c1 = t.tets_batch()
        t.clear()
        t.batch(xd, off)
        again, c2 = t.tets_batch()
        st = t.stats()
        assert st["batch_graph"] == 1
        assert np.array_equal(first, again) and np.array_equal(c1, c2)
        xyz2 = synth.uniform(99, 3 * len(xyz)).reshape(-1, 3)  # same cloud sizes, new coordinates
        xd.copy_(torch.from_numpy(xyz2 * 3.0 - 1.0))
        t.clear()
        t.batch(xd, off)
        new, c3 = t.tets_batch()
        assert t.stats()["batch_graph"] == 1
    clouds = split(xyz2 * 3.0 - 1.0, off)
    assert_clouds_match(clouds, [new[int(c3[c]):int(c3[c + 1])] for c in range(30)])


@pytest.mark.parametrize("subdet", [False, True])
def test_insert_after_a_larger_batch_on_the_same_handle(subdet, monkeypatch):
    """A batch grows the tetrahedron store, its owner words and its free list, but not the
    sub-determinant cache: an insert that follows on the handle has to bring an entry per slot."""
    if subdet:
        monkeypatch.setenv("DT_SUBDET", "1")
    xyz, off = synth.batched_clouds(12, 5, lo=50, hi=3000)
    x = synth.uniform_cube(900, 6)
    small = synth.uniform_cube(60, 7)
    ref, _ = oracle.delaunay(x)
    for first in (None, small):  # without a cache yet, and with one shorter than the batch's store
        with dt.Triangulation(seed=0) as t:
            if first is not None:
                t.insert(torch.from_numpy(first).cuda())
            grown = []
            for _ in range(2):
                t.batch(torch.from_numpy(xyz).cuda(), off)
                before = t.stats()["device_bytes"]
                t.clear()
                t.insert(torch.from_numpy(x).cuda())
                assert np.array_equal(t.tets_numpy(), ref)
                grown.append(t.stats()["device_bytes"] - before)
            # an entry of 32 bytes for each of the store's slots (8 a point at least, all but the
            # 6000 the first insert may have brought)
            assert not subdet or grown[0] >= 32 * (8 * len(xyz) - 6000) > 0


@pytest.mark.parametrize("sizes", [(0, 3, 4, 5, 6), (2047, 2048, 2049), (14336, 14337, 40), (1,), (900, 20001)])
def test_batch_at_the_edges_of_waves_and_segments(sizes):
    """Cloud sizes around the BRIO round ends, clouds with nothing to insert, and a cloud whose
    launches go on long after the others' last wave."""
    clouds = [synth.uniform_cube(n, 300 + n) if n else np.zeros((0, 3)) for n in sizes]
    if sizes == (1,):
        with pytest.raises(dt.DTError) as e:
            run_batch(clouds)
        assert e.value.code == dt.DT_EDEGENERATE
        return
    got, st = run_batch(clouds)
    assert st["n_clouds_degenerate"] == sum(n < 4 for n in sizes)
    for c, x in enumerate(clouds):
        ref = oracle.delaunay(x)[0] if len(x) >= 4 else np.zeros((0, 4), np.uint32)
        assert np.array_equal(got[c], ref), c


def test_batch_cavities_beyond_the_borrowed_workspaces():
    """Centres of shells: cavities of hundreds to thousands of tetrahedra, in the borrowed and in the
    largest workspaces, beside an ordinary cloud."""
    g = np.random.default_rng(5)
    clouds = [synth.uniform_cube(500, 6)]
    for n in (300, 3000):
        s = g.normal(size=(n, 3))
        s /= np.linalg.norm(s, axis=1, keepdims=True)
        clouds.append(np.concatenate([s, 0.01 * g.normal(size=(5, 3))]))
    got, _ = run_batch(clouds)
    assert_clouds_match(clouds, got)


def test_batch_refuses_bad_coordinates_and_goes_on():
    xyz, off = synth.batched_clouds(6, 8, lo=50, hi=500)
    bad = xyz.copy()
    bad[77, 1] = np.nan
    with dt.Triangulation(seed=0) as t:
        for _ in range(2):
            with pytest.raises(dt.DTError) as e:
                t.batch(torch.from_numpy(bad).cuda(), off)
            assert e.value.code == dt.DT_EINVAL
        t.clear()
        t.batch(torch.from_numpy(xyz).cuda(), off)
        tets, coff = t.tets_batch()
    assert_clouds_match(split(xyz, off), [tets[int(coff[c]):int(coff[c + 1])] for c in range(6)])


@pytest.mark.parametrize("earlier", [0, 2, 40])
def test_no_rows_after_a_refused_batch(earlier):
    """The list between a refused batch and the clear: no rows, on a fresh handle and after smaller
    and larger batches, through every form of the list."""
    xyz, off = synth.batched_clouds(6, 8, lo=50, hi=500)
    bad = xyz.copy()
    bad[77, 1] = np.inf
    with dt.Triangulation(seed=0) as t:
        if earlier:
            x0, off0 = synth.batched_clouds(earlier, 9, lo=50, hi=300)
            t.batch(torch.from_numpy(x0).cuda(), off0)
        with pytest.raises(dt.DTError) as e:
            t.batch(torch.from_numpy(bad).cuda(), off)
        assert e.value.code == dt.DT_EINVAL
        out = torch.zeros((9000, 4), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
        for canonical in (True, False):
            assert len(t.tets_host(canonical=canonical, out=out)) == 0
            for buf in (out, None):
                rows, coff = t.tets_batch(canonical=canonical, out=buf)
                assert len(rows) == 0 and coff.shape == (7,) and not coff.any()
        assert t.num_tets() == 0 and not out.any()
        t.batch(torch.from_numpy(xyz).cuda(), off)
        tets, coff = t.tets_batch()
        assert np.array_equal(t.tets_host(), tets)
        with pytest.raises(dt.DTError):  # refused arguments: the last batch stays
            t.batch(torch.from_numpy(xyz).cuda(), off[::-1].copy())
        again, coff2 = t.tets_batch()
        assert np.array_equal(again, tets) and np.array_equal(coff2, coff)
    assert_clouds_match(split(xyz, off), [tets[int(coff[c]):int(coff[c + 1])] for c in range(6)])


@pytest.mark.parametrize("steps", [1, 8])
def test_batch_of_needles_with_short_walks(steps):
    """Walks of hundreds of steps (the hint cells of a thin cloud hold whole slices of it): a short
    max_walk_steps leaves no point behind, and takes no other time than the default."""
    g = np.random.default_rng(1)
    clouds = [g.random((n, 3)) * (1.0, thin, thin) for n, thin in ((3000, 1e-3), (3000, 1e-6), (20000, 1e-3))]
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    ms = []
    for limit in (0, steps):
        with dt.Triangulation(seed=0, max_walk_steps=limit) as t:
            t.batch(x, np.array([0, 3000, 6000, 26000]))
            tets, coff = t.tets_batch()
            ms.append(t.stats()["ms_insert"])
        assert_clouds_match(clouds, [tets[int(coff[c]):int(coff[c + 1])] for c in range(3)])
    assert ms[1] < 5 * ms[0]  # 300 times when every launch stopped the walks


def test_an_empty_cloud_does_not_widen_the_others_error_bounds():
    """The FP32 stage's error term comes from the largest coordinate of the batch; with an empty
    cloud's infinite box in it, no test of any cloud was decided in FP32 (2.2 times the time)."""
    clouds = [synth.uniform_cube(n, n) for n in (2000, 3000, 500)]
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    best = []
    for off in ([0, 2000, 5000, 5500], [0, 0, 2000, 5000, 5000, 5500, 5500]):
        with dt.Triangulation(seed=0) as t:
            ms = []
            for _ in range(8):
                t.batch(x, np.array(off))
                ms.append(t.stats()["ms_insert"])
            tets, coff = t.tets_batch()
        best.append(min(ms))
        got = [tets[int(coff[c]):int(coff[c + 1])] for c in range(len(off) - 1) if off[c + 1] > off[c]]
        assert_clouds_match(clouds, got)
    assert best[1] < 1.5 * best[0]


def test_many_clouds_take_no_more_memory_than_their_points_need():
    """The store is 60 bytes for each of 8 slots a point, 64 a cloud, and 64 for each warp that a
    cloud is planned to have: a hundredth of its points when many clouds fill the device (an eighth
    more slots, where the warps it would have alone made it 2.2 times the points' share)."""
    xyz, off = synth.batched_clouds(2000, 4, lo=50, hi=2000)
    with dt.Triangulation(seed=0) as t:
        t.batch(torch.from_numpy(xyz).cuda(), off)
        held = t.stats()["device_bytes"]
    points = 220 * len(xyz)  # records, order, lists: bytes a point beside the store's
    assert held < points + 1.5 * 60 * (8 * len(xyz) + 64 * 2000)


def test_statistics_cover_the_launches_after_the_planned_ones():
    """Cavities of up to 6000 tetrahedra are inserted by launches after the planned sequence: they
    count as large cavities and as launches, and their time is in ms_insert."""
    g = np.random.default_rng(5)
    s = g.normal(size=(6000, 3))
    shell = np.concatenate([s / np.linalg.norm(s, axis=1, keepdims=True), 0.01 * g.normal(size=(5, 3))])
    seen = {}
    for name, x in (("plain", synth.uniform_cube(len(shell), 3)), ("shell", shell)):
        xd, off = torch.from_numpy(x).cuda(), np.array([0, len(x)])
        with dt.Triangulation(seed=0) as t:
            share = []  # of the call's time that the statistics account for
            for _ in range(6):
                torch.cuda.synchronize()
                begin = time.perf_counter()
                t.batch(xd, off)
                wall = 1e3 * (time.perf_counter() - begin)
                seen[name] = t.stats()
                share.append((seen[name]["ms_sort"] + seen[name]["ms_insert"]) / wall)
        assert max(share) > 0.6, share  # the best of them: the host may be busy
        assert seen[name]["batch_min_blocks"] == 4
    assert seen["shell"]["n_rounds"] > seen["plain"]["n_rounds"]
    # one at least: without a cavity beyond the borrowed workspaces there are no such launches
    assert 1 <= seen["shell"]["n_big"] <= len(shell)
    xyz, off = synth.batched_clouds(1500, 4, lo=500, hi=5000)  # more than 2432 segments in a launch
    with dt.Triangulation(seed=0) as t:
        t.batch(torch.from_numpy(xyz).cuda(), off)
        assert t.stats()["batch_min_blocks"] == 6
