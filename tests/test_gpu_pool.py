"""The pooled search (traversal variant 0, and every width of several lanes per query)
against the one-thread search of the same queries: bit for bit, at the edges of its
warps, with its stack nearly full and with more tied faces than a query records."""
import numpy as np
import pytest
import torch

from paper_2606_00444_gb300 import MeshBatch, MeshBVH
from parity import assert_identical, dev
from workloads.meshes import displaced_icosphere, icosphere
from workloads.sampling import uniform_box

pytestmark = pytest.mark.gpu

LANES = [1, 2, 4, 8, 16, 32]


def one_thread(bvh, Q, md, hint=None):
    bvh.set_query_config(1, 2)
    out = bvh.closest_point(Q, md, hint=hint)
    bvh.set_query_config(-1, -1)
    return out


def pooled(bvh, Q, md, lanes, hint=None):
    bvh.set_query_config(lanes, 0)
    out = bvh.closest_point(Q, md, hint=hint)
    bvh.set_query_config(-1, -1)
    return out


@pytest.mark.parametrize("lanes", LANES)
@pytest.mark.parametrize("faces", [1, 2, 3, 1280])
def test_ragged_query_counts(lanes, faces):
    V, F = displaced_icosphere(3, 0.1, 0.4)
    F = np.ascontiguousarray(F[:faces])
    bvh = MeshBVH.from_mesh(dev(V), dev(F))
    S = 32 // lanes
    for n in sorted({1, S - 1, S, S + 1, 3 * S + 1, 67}):
        if n < 1:
            continue
        Q = dev(uniform_box(n, [-1.5] * 3, [1.5] * 3, seed=n))
        for md in (float("inf"), 0.3, 0.0):
            ref = one_thread(bvh, Q, md)
            assert_identical(pooled(bvh, Q, md, lanes), ref)
            assert_identical(pooled(bvh, Q, md, lanes, hint=ref["face"]), ref)
    assert bvh.status()[0] == 0


@pytest.mark.parametrize("method", ["lbvh", "ploc"])
@pytest.mark.parametrize("lanes", LANES)
def test_deep_searches_with_the_stack_nearly_full(lanes, method):
    """Queries about the centre of a sphere: every face is nearly equally near, so each
    search defers a sibling at almost every level of the tree."""
    V, F = icosphere(5)
    bvh = MeshBVH.from_mesh(dev(V), dev(F), method=method)
    rng = np.random.default_rng(5)
    Q = dev((rng.normal(size=(64, 3)) * 1e-3).astype(np.float32))
    ref = one_thread(bvh, Q, float("inf"))
    assert_identical(pooled(bvh, Q, float("inf"), lanes), ref)
    ref = one_thread(bvh, Q, 1.5)                         # a cutoff that prunes nothing: the shallow stacks
    assert_identical(pooled(bvh, Q, 1.5, lanes), ref)
    assert bvh.status()[0] == 0


@pytest.mark.parametrize("lanes", LANES)
@pytest.mark.parametrize("leaf", [1, 4])
def test_more_tied_faces_than_a_query_records(lanes, leaf):
    """A fan of 40 faces around one vertex, queried at and above it, and a stack of 40
    copies of one face: all are at the same distance, the lowest id wins."""
    t = np.linspace(0, 2 * np.pi, 40, endpoint=False)
    V = np.concatenate([[[0, 0, 1]], np.stack([np.cos(t), np.sin(t), 0 * t], 1)]).astype(np.float32)
    i = np.arange(40)
    fan = np.stack([0 * i, 1 + i, 1 + (i + 1) % 40], 1).astype(np.int32)
    rng = np.random.default_rng(1)
    for F in (fan[rng.permutation(40)], np.repeat(fan[:1], 40, 0)):
        bvh = MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(F)))
        bvh.set_leaf_size(leaf)
        Q = dev(np.array([[0, 0, 1], [0, 0, 2], [0, 0, 1.001], [0.1, 0.2, 3]], np.float32))
        for md in (float("inf"), 2.5):
            assert_identical(pooled(bvh, Q, md, lanes), one_thread(bvh, Q, md))
        assert int(pooled(bvh, Q, float("inf"), lanes)["face"][1]) == 0
        assert bvh.status()[0] == 0


def test_batch_warps_that_span_scenes():
    """Scenes of a few queries each, some with no faces: one warp holds queries of many."""
    rng = np.random.default_rng(9)
    meshes, qs = [], []
    for k in range(23):
        V, F = displaced_icosphere(int(rng.integers(0, 4)), 0.1, 0.1 * k)
        V = (V * rng.uniform(0.1, 50.0)).astype(np.float32)
        F = F[:[0, 1, 2, len(F)][k % 4]]
        meshes.append((V, np.ascontiguousarray(F)))
        qs.append(uniform_box(int(rng.integers(0, 9)), V.min(0) * 1.2, V.max(0) * 1.2, seed=k))
    batch = MeshBatch.from_meshes(meshes)
    off = dev(np.concatenate([[0], np.cumsum([len(q) for q in qs])]).astype(np.int32))
    for md in (float("inf"), 0.5):
        got = batch.closest_point(dev(np.concatenate(qs)), off, md)
        ref = [one_thread(MeshBVH.from_mesh(dev(v), dev(f)), dev(q), md) for (v, f), q in zip(meshes, qs) if len(q)]
        assert_identical(got, {k: torch.cat([r[k] for r in ref]) for k in ref[0]})
    assert batch.status()[0] == 0


@pytest.mark.parametrize("n", [1, 3, 33, 100_003])
@pytest.mark.parametrize("k,leaf", [(1, 1), (4, 1), (8, 1), (8, 4)])
def test_knn_lists_are_the_k_least_distances(n, k, leaf):
    """The k faces of each query, checked against every face's own distance (a mesh of that
    face alone): the k least, nearest first, with the lower id first among equals; at the
    pooled widths 1-8 (by the query count), meshes smaller than k, and leaf ranges."""
    V, F = icosphere(1)
    rng = np.random.default_rng(n + k)
    Qn = (rng.normal(size=(n, 3))).astype(np.float32)
    Qn[: min(n, 12)] = V[: min(n, 12)]                    # on vertices: ties of five faces
    for faces in (3, len(F)):
        Fs = np.ascontiguousarray(F[:faces])
        bvh = MeshBVH.from_mesh(dev(V), dev(Fs))
        bvh.set_leaf_size(leaf)
        _, face, d2 = bvh.knn_project(dev(Qn), k=k, want_faces=True)
        m = min(n, 200)
        Q = dev(Qn[:m])
        each = torch.stack([one_thread(MeshBVH.from_mesh(dev(V), dev(Fs[f:f + 1])), Q, float("inf"))["dist2"]
                            for f in range(faces)], 1).cpu().numpy()
        order = np.lexsort((np.broadcast_to(np.arange(faces), each.shape), each), axis=1)[:, :k]
        c = min(k, faces)
        assert np.array_equal(face[:m, :c].cpu().numpy(), order)
        assert np.array_equal(d2[:m, :c].cpu().numpy(), np.take_along_axis(each, order, 1))
        assert (face[:, c:] == -1).all() and torch.isinf(d2[:, c:]).all()
        assert bvh.status()[0] == 0


@pytest.mark.parametrize("lanes", LANES)
@pytest.mark.parametrize("leaf", [1, 4])
def test_fronts_of_falling_ids_over_rising_distances(lanes, leaf):
    """Layers of faces one float32 step apart, the nearer ones with the higher ids: up to 17
    of them lie inside a tie window and none rules out another, more than the rings of 8, 12
    and 16 hold (the search is then decided by resolve_ties); with the ids in no order a few
    remain.  Each layer is three copies, so that many faces are met at once."""
    base = np.float32(0.99999)
    z = -(base + np.arange(40, dtype=np.float32) * np.float32(2.0 ** -24))
    V = np.stack([[[-9, -9, h], [9, -9, h], [0, 9, h]] for h in z]).reshape(-1, 3).astype(np.float32)
    layers = np.arange(120, dtype=np.int32).reshape(40, 3)
    rng = np.random.default_rng(2)
    falling = np.repeat(layers[::-1], 3, 0)               # the nearest layer last
    for F in (falling, falling[rng.permutation(120)]):
        bvh = MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(F)))
        bvh.set_leaf_size(leaf)
        Q = np.zeros((70, 3), np.float32)
        Q[:, :2] = rng.uniform(-1, 1, (70, 2))
        Q[::2, 2] = rng.uniform(0, 1, 35)
        for md in (float("inf"), 1.5):
            assert_identical(pooled(bvh, dev(Q), md, lanes), one_thread(bvh, dev(Q), md))
        assert bvh.status()[0] == 0


def _best_ms(fn, repeats=12):
    fn()
    ts = []
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return min(ts)


def test_tied_faces_are_not_left_to_one_lane():
    """From 1000 radii away hundreds of faces of a sphere lie inside the tie window: 100 such
    queries take at most 4 times as long as 100 from 3 radii (they meet more faces; with the
    ties left to one lane's search they took 11 times as long)."""
    V, F = icosphere(6)
    bvh = MeshBVH.from_mesh(dev(V), dev(F))
    d = np.random.default_rng(0).normal(size=(100, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    ms = []
    for r in (3.0, 1000.0):
        Q = dev((d * r).astype(np.float32))
        out = bvh.closest_point(Q)
        assert_identical(out, one_thread(bvh, Q, float("inf")))
        ms.append(_best_ms(lambda: bvh.closest_point(Q, out=out)))
    assert ms[1] <= 4 * ms[0], ms


@pytest.mark.parametrize("n", [100, 50_000])
@pytest.mark.parametrize("signed", [False, True])
def test_loose_cutoffs_cost_no_more_than_none(n, signed):
    """A cutoff that every query's answer meets by far prunes nothing by itself: the search
    takes at most 1.5 times the time of the one without a cutoff (it took 3 to 20 times as
    long when it started without a radius)."""
    V, F = icosphere(6)
    bvh = MeshBVH.from_mesh(dev(V), dev(F))
    rng = np.random.default_rng(n)
    Q = dev((V[rng.integers(0, len(V), n)] + rng.normal(size=(n, 3)) * 0.02).astype(np.float32))
    find = bvh.signed_distance if signed else bvh.closest_point
    ref = find(Q)
    free_ms = _best_ms(lambda: find(Q, out=ref))
    for md in (0.3, 0.7, 2.0):
        got = find(Q, md)
        assert_identical(got, ref)
        assert _best_ms(lambda: find(Q, md, out=got)) <= 1.5 * free_ms


def test_searches_under_a_cutoff_from_wherever_they_start():
    """Cutoffs from none of the mesh to all of it (the search starts at the first node with two
    children inside, or ends there; a loose cutoff first goes down to a leaf), with and
    without hints and leaf ranges: the one-thread search's answers."""
    V, F = displaced_icosphere(4, 0.1, 0.4)
    for faces, leaf in ((len(F), 1), (len(F), 4), (2, 1), (3, 4)):
        bvh = MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(F[:faces])))
        bvh.set_leaf_size(leaf)
        Q = dev(np.concatenate([uniform_box(3000, [-1.5] * 3, [1.5] * 3, seed=4), np.full((3, 3), 1e6)]).astype(np.float32))
        for md in (0.0, 1e-3, 0.02, 0.1, 0.3, 1.0, 5.0, 1e9):
            ref = one_thread(bvh, Q, md)
            for lanes in (-1, 2, 32):
                assert_identical(pooled(bvh, Q, md, lanes), ref)
                assert_identical(pooled(bvh, Q, md, lanes, hint=ref["face"]), ref)


@pytest.mark.parametrize("faces", [1, 2, 16, 17, 24, 25])
def test_meshes_of_few_faces(faces):
    """Up to 16 faces (24 with many queries) a thread per query tests them all: closest points,
    signed distances and Chamfer samples equal the one-thread search's, faces tied or not."""
    from paper_2606_00444_gb300 import chamfer
    V, F = displaced_icosphere(1, 0.1, 0.4)
    F = np.ascontiguousarray(F[:faces])
    for Fm in (F, np.repeat(F[:1], faces, 0)):
        bvh = MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(Fm)))
        for n in (1, 127, 129, 50_001):
            Q = dev(uniform_box(n, [-1.5] * 3, [1.5] * 3, seed=n))
            for md in (float("inf"), 0.5, 0.0):
                ref = one_thread(bvh, Q, md)
                assert_identical(bvh.closest_point(Q, md), ref)
                assert_identical(bvh.signed_distance(Q, md), ref)
            out, ps = chamfer(bvh, Q, bvh, Q, per_sample=True)
            ref = one_thread(bvh, Q, float("inf"))
            assert torch.equal(ps["faceA"], ref["face"]) and torch.equal(ps["dist2B"], ref["dist2"])
            assert torch.allclose(out, ref["dist2"].double().mean().expand(2), rtol=1e-12)
        assert bvh.status()[0] & ~8 == 0                   # (8: copies of a face are no manifold)


def test_batch_of_mostly_few_faces():
    """Scenes of few faces on average, some of them large, some without faces: warps
    that hold queries of several of each."""
    rng = np.random.default_rng(3)
    meshes, qs = [], []
    for k in range(60):
        V, F = displaced_icosphere(2 if k == 7 else 1, 0.1, 0.1 * k)
        V = (V * rng.uniform(0.1, 50.0)).astype(np.float32)
        F = F if k == 7 else F[:[1, 0, 5, 24, 25][k % 5]]
        meshes.append((V, np.ascontiguousarray(F)))
        qs.append(uniform_box(int(rng.integers(0, 40)), V.min(0) * 1.2, V.max(0) * 1.2, seed=k))
    batch = MeshBatch.from_meshes(meshes)
    assert sum(len(f) for _, f in meshes) <= 17 * len(meshes) and max(len(f) for _, f in meshes) == 320
    off = dev(np.concatenate([[0], np.cumsum([len(q) for q in qs])]).astype(np.int32))
    for md in (float("inf"), 0.5):
        got = batch.closest_point(dev(np.concatenate(qs)), off, md)
        ref = [one_thread(MeshBVH.from_mesh(dev(v), dev(f)), dev(q), md) for (v, f), q in zip(meshes, qs) if len(q)]
        assert_identical(got, {k: torch.cat([r[k] for r in ref]) for k in ref[0]})
    assert batch.status()[0] == 0


def test_few_faces_cost_no_more_than_one_thread_per_query():
    """300k queries of meshes of one and of four faces, and 300k Chamfer samples a side: at most
    1.3 times the one-thread search's time for as many queries (a warp of the pool per 16
    samples: twice)."""
    from paper_2606_00444_gb300 import Workspace, chamfer
    V, F = icosphere(1)
    Q = dev(uniform_box(300_000, [-1.5] * 3, [1.5] * 3, seed=1))
    for faces in (1, 4):
        bvh = MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(F[:faces])))
        ref = one_thread(bvh, Q, float("inf"))
        bvh.set_query_config(1, 2)
        one_ms = _best_ms(lambda: bvh.closest_point(Q, out=ref))
        bvh.set_query_config(-1, -1)
        got = bvh.closest_point(Q)
        assert _best_ms(lambda: bvh.closest_point(Q, out=got)) <= 1.3 * one_ms
        ws, cd = Workspace(Q.device), torch.empty(2, dtype=torch.float64, device="cuda")
        assert _best_ms(lambda: chamfer(bvh, Q, bvh, Q, ws=ws, out=cd)) <= 1.3 * 2 * one_ms


@pytest.mark.parametrize("faces", [1, 3, 16, 17, 24, 25])
@pytest.mark.parametrize("n", [1, 33, 50_001])
def test_knn_of_few_or_tied_faces(n, faces):
    """Meshes of few faces (a lane per query tests them all) and many tied faces (copies, at
    a query's own distance): the lists are the k least (distance, id)."""
    V, F = icosphere(1)
    rng = np.random.default_rng(n)
    Qn = rng.normal(size=(n, 3)).astype(np.float32)
    Qn[0] = 0.0
    for Fs in (F[:faces], np.concatenate([F[:faces], F[:faces][::-1]])):
        Fs = np.ascontiguousarray(Fs)
        bvh = MeshBVH.from_mesh(dev(V), dev(Fs))
        m = min(n, 100)
        each = torch.stack([one_thread(MeshBVH.from_mesh(dev(V), dev(Fs[f:f + 1])), dev(Qn[:m]), float("inf"))["dist2"]
                            for f in range(len(Fs))], 1).cpu().numpy()
        order = np.lexsort((np.broadcast_to(np.arange(len(Fs)), each.shape), each), axis=1)
        for k in (1, 4, 8):
            p, face, d2 = bvh.knn_project(dev(Qn), k=k, want_faces=True)
            c = min(k, len(Fs))
            assert np.array_equal(face[:m, :c].cpu().numpy(), order[:, :c])
            assert np.array_equal(d2[:m, :c].cpu().numpy(), np.take_along_axis(each, order[:, :c], 1))
            assert (face[:, c:] == -1).all() and torch.isinf(d2[:, c:]).all() and torch.isfinite(p).all()
        assert bvh.status()[0] == 0


def test_knn_of_tied_faces_costs_no_more_than_the_nearest():
    """50k queries at the centre of a cube whose sides are 8 nearest faces each: the nearest face
    by k-NN takes at most 3 times the unbounded closest point's time (inserting every
    tied face took 5 times); of 4 faces, the 4 nearest at most 3 times (9)."""
    g = np.arange(41)
    u, v = (x.ravel() for x in np.meshgrid(g, g, indexing="ij"))
    i, j = (x.ravel() for x in np.meshgrid(g[:-1], g[:-1], indexing="ij"))
    q = [(i + a) * 41 + j + b for a, b in ((0, 0), (1, 0), (1, 1), (0, 1))]
    side = np.concatenate([np.stack([q[0], q[1], q[2]], 1), np.stack([q[0], q[2], q[3]], 1)])
    V = np.concatenate([np.roll(np.stack([u / 20 - 1, v / 20 - 1, 0 * u + s], 1), k, axis=1)
                        for k in range(3) for s in (-1.0, 1.0)]).astype(np.float32)
    F = np.concatenate([side + 1681 * k for k in range(6)]).astype(np.int32)
    Vs, Fs = icosphere(1)
    for (Vm, Fm, k, n) in ((V, F, 1, 50_000), (Vs, np.ascontiguousarray(Fs[:4]), 4, 300_000)):
        bvh = MeshBVH.from_mesh(dev(Vm), dev(Fm))
        Q = torch.zeros(n, 3, device="cuda")
        out, p = bvh.closest_point(Q), bvh.knn_project(Q, k=k)
        cp_ms = _best_ms(lambda: bvh.closest_point(Q, out=out))
        assert _best_ms(lambda: bvh.knn_project(Q, k=k, out=p)) <= 3 * cp_ms


@pytest.mark.parametrize("n", [6_000, 25_000, 50_000, 100_000, 200_000])
def test_batch_warps_of_every_width_span_scenes(n):
    """Widths of 1, 2, 4, 8 and 16 queries per warp (by the query count) over 300 scenes of
    different sizes and scales, some without faces or without queries."""
    rng = np.random.default_rng(n)
    meshes, qs = [], []
    for k in range(300):
        V, F = displaced_icosphere(int(rng.integers(1, 4)), 0.1, 0.1 * k)
        V = (V * rng.uniform(0.1, 50.0) + rng.uniform(-5, 5, 3)).astype(np.float32)
        F = F[:0] if k % 17 == 5 else F
        meshes.append((V, np.ascontiguousarray(F)))
        m = 0 if k % 11 == 3 else int(rng.integers(0, n // 136))
        qs.append(uniform_box(m, V.min(0) - 0.1, V.max(0) + 0.1, seed=k))
    batch = MeshBatch.from_meshes(meshes)
    off = dev(np.concatenate([[0], np.cumsum([len(q) for q in qs])]).astype(np.int32))
    Q = dev(np.concatenate(qs))
    singles = [MeshBVH.from_mesh(dev(v), dev(f)) for v, f in meshes]
    for md in (float("inf"), 0.5):
        got = batch.closest_point(Q, off, md)
        ref = [one_thread(b, dev(q), md) for b, q in zip(singles, qs) if len(q)]
        assert_identical(got, {k: torch.cat([r[k] for r in ref]) for k in ref[0]})
    assert batch.status()[0] == 0


@pytest.mark.parametrize("n", [25_003, 50_003])
@pytest.mark.parametrize("k,leaf", [(4, 1), (8, 4)])
def test_knn_of_two_and_four_queries_per_warp(n, k, leaf):
    V, F = icosphere(1)
    bvh = MeshBVH.from_mesh(dev(V), dev(F))
    bvh.set_leaf_size(leaf)
    Qn = np.random.default_rng(n + k).normal(size=(n, 3)).astype(np.float32)
    Qn[:12] = V[:12]                                      # on vertices: ties of five faces
    pick = np.r_[0:100, n - 100:n]
    p, face, d2 = bvh.knn_project(dev(Qn), k=k, want_faces=True)
    Q = dev(Qn[pick])
    each = torch.stack([one_thread(MeshBVH.from_mesh(dev(V), dev(np.ascontiguousarray(F[f:f + 1]))), Q, float("inf"))["dist2"]
                        for f in range(len(F))], 1).cpu().numpy()
    order = np.lexsort((np.broadcast_to(np.arange(len(F)), each.shape), each), axis=1)[:, :k]
    assert np.array_equal(face.cpu().numpy()[pick], order)
    assert np.array_equal(d2.cpu().numpy()[pick], np.take_along_axis(each, order, 1))
    assert torch.isfinite(p).all() and bvh.status()[0] == 0


def test_chamfer_of_32_samples_per_warp():
    """mesh_chamfer_noalloc with more samples than its scratch holds blocks of 64 for: 32 queries
    per warp, the per-sample results of mesh_chamfer."""
    from paper_2606_00444_gb300 import chamfer
    from paper_2606_00444_gb300._abi import check, lib
    V, F = displaced_icosphere(3, 0.1, 0.4)
    bvh = MeshBVH.from_mesh(dev(V), dev(F))
    nA, nB = 600_011, 500_003
    assert (nA + nB) * 2 > 16384 * 128 > nA + nB
    SA, SB = (dev(uniform_box(n, [-1.2] * 3, [1.2] * 3, seed=n)) for n in (nA, nB))
    ref, ps = chamfer(bvh, SA, bvh, SB, per_sample=True)
    out = torch.empty(2, dtype=torch.float64, device="cuda")
    got = {k: torch.empty_like(v) for k, v in ps.items()}
    check(lib().mesh_chamfer_noalloc(bvh.handle, SA.data_ptr(), nA, bvh.handle, SB.data_ptr(), nB, out.data_ptr(),
                                     *(got[k].data_ptr() for k in ("faceA", "baryA", "dist2A", "faceB", "baryB", "dist2B")),
                                     torch.cuda.current_stream().cuda_stream), "mesh_chamfer_noalloc")
    for k in ps:
        assert torch.equal(got[k], ps[k]), k
    assert torch.allclose(out, ref, rtol=1e-12)
