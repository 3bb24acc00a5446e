"""GPU parity of the scheduler where its kernels change form: one warp per matrix (up to four groups of four) in 32-bit granules
and in bytes, one and two lanes per rank group, tasks of a part of a warp up to two warps, scores within and beyond 32 bits,
other numbers of starts and sweeps than four and three, plans cut short."""
import itertools

import numpy as np
import pytest
import torch

import tests.test_gpu_schedule as ts
from tests.test_gpu_schedule import vp  # noqa: F401  (fixture)
from workloads import SchedParams as WParams, complete_catalog, node_template_catalog, tree_topology
from workloads.topology import Catalog, _assemble, ring_topology

pytestmark = pytest.mark.gpu

CATALOGS = {
    "one_node": lambda: complete_catalog(tree_topology(1)),
    "ring_of_three": lambda: complete_catalog(ring_topology(1, switches_per_node=3, g=4)),
    "two_nodes_64_50": lambda: complete_catalog(tree_topology(2, nic_bw=50)),
    "template_1": lambda: node_template_catalog(tree_topology(1)),
    "template_3_64_50": lambda: node_template_catalog(tree_topology(3, nic_bw=50)),
    "template_4": lambda: node_template_catalog(tree_topology(4)),
    "template_5_64_50": lambda: node_template_catalog(tree_topology(5, nic_bw=50)),
    "template_8": lambda: node_template_catalog(tree_topology(8)),
    "template_9": lambda: node_template_catalog(tree_topology(9)),
    "template_17": lambda: node_template_catalog(tree_topology(17)),
}


@pytest.mark.parametrize("name", sorted(CATALOGS))
def test_magnitudes_starts_and_sweeps(vp, oracle_lib, name):  # noqa: F811
    cat = CATALOGS[name]()
    N = cat.topology.N
    rng = np.random.default_rng(len(name) + N)
    B = 6
    # largest entry (granules of 256 bytes): ordinary, beyond 16 bits, scores beyond 32 bits, capacities beyond 2^22 granules
    for hi, kt, n_start, i_aa, k_max in [(900, 2 * N, 4, 3, 10 * N), (70000, N, 3, 2, 10 * N), (1 << 24, 2 * N, 4, 1, 10 * N),
                                         ((1 << 32) - 1, 8, 4, 3, 40), (5000, N, 5, 4, N // 2), (300, 3 * N, 1, 3, 10 * N)]:
        D = rng.integers(0, hi + 1, size=(B, N, N)) * (rng.random((B, N, N)) < (0.6 if N < 64 else 0.15)) * 256
        D[1] = 0
        D[2] //= 512
        D[2] *= 256
        D[3][:, 0] = hi * 256                                  # one popular destination
        for b in range(B):
            np.fill_diagonal(D[b], 0)
        w = WParams(granule_bytes=256, k_target=kt, n_start=n_start, i_aa=i_aa, k_max=k_max).resolved(N)
        got, want, *_ = ts._both(vp, oracle_lib, cat, D.astype(np.int64), w)
        ts._assert_same(got, want)


@pytest.mark.parametrize("name,batches", [("one_node", (1, 593, 1185)), ("two_nodes_64_50", (1, 593, 1185)), ("template_8", (296, 297, 593)),
                                          ("template_5_64_50", (593, 700)), ("template_9", (149, 297))])
def test_work_counters_and_batches(vp, oracle_lib, name, batches):  # noqa: F811
    """Batches on both sides of the launch shapes' limits give the same plans, and the work counters add up."""
    import torch
    cat = CATALOGS[name]()
    N = cat.topology.N
    rng = np.random.default_rng(N)
    base = (rng.integers(0, 60, size=(3, N, N)) * (rng.random((3, N, N)) < 0.5) * 4096).astype(np.int64)
    for b in range(3):
        np.fill_diagonal(base[b], 0)
    w = WParams(granule_bytes=4096).resolved(N)
    oc = oracle_lib.OracleCatalog(cat.topology.blob(), cat.blob())
    dc = vp.load_catalog(cat.topology.blob(), cat.blob())
    want = oc.schedule_batch(base, w, threads=3)
    p = ts._params(vp, w)
    for B in batches:
        D = torch.from_numpy(np.tile(base, ((B + 2) // 3, 1, 1))[:B].copy()).cuda()
        ws = torch.full((vp.schedule_workspace_bytes(dc, B, p),), 0x5A, dtype=torch.uint8, device="cuda")
        got = vp.schedule_batch(dc, p, D, workspace=ws)
        stats = vp.schedule_read_stats(ws)
        got = got.cpu()
        for key in ts.KEYS:
            for r in range(0, B, 3):
                n = min(3, B - r)
                assert np.array_equal(got[key][r:r + n], want[key][:n]), (B, key, r)
        assert stats["activations"] == int(got["n_steps"].sum()) and stats["tasks"] >= 4 * stats["activations"] and stats["sweeps"] >= stats["tasks"]


@pytest.mark.parametrize("name,B", [("two_nodes_64_50", 70), ("template_5_64_50", 7), ("template_8", 5), ("template_17", 3)])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_rows_in_use(vp, oracle_lib, name, B, pinned):  # noqa: F811
    """Rows in use come back the same through page-locked buffers (written by the scheduler) and pageable ones (copied), with
    receive offsets and without a matrix's idle rows being touched; one invalid matrix, one cut short."""
    import torch
    cat = CATALOGS[name]()
    N = cat.topology.N
    rng = np.random.default_rng(B)
    D = (rng.integers(0, 90, size=(B, N, N)) * (rng.random((B, N, N)) < (0.5 if N < 64 else 0.1)) * 512).astype(np.int64)
    D[0] *= (rng.random((N, N)) < 0.05)
    for b in range(B):
        np.fill_diagonal(D[b], 0)
    D[1, 3, 3] = 512
    w = WParams(granule_bytes=512, k_max=3 * N).resolved(N)
    oc = oracle_lib.OracleCatalog(cat.topology.blob(), cat.blob())
    dc = vp.load_catalog(cat.topology.blob(), cat.blob())
    p = ts._params(vp, w)
    plan = vp.Plan.empty(B, N, p.k_max, "cpu", pin=pinned)
    for key in ("chan_id", "lane_dst", "lane_inst", "lane_bytes", "send_off", "recv_off"):
        getattr(plan, key).fill_(77)
    demand = torch.from_numpy(D)
    vp.schedule_batch_host(dc, p, demand.pin_memory() if pinned else demand, plan=plan, used_only=True)
    want, got = oc.schedule_batch(D, w, threads=B), plan.cpu()
    for key in ("n_steps", "status", "tau_ns"):
        assert np.array_equal(got[key], want[key]), key
    for b in range(B):
        K = int(want["n_steps"][b])
        for key, n in (("chan_id", K), ("lane_dst", K), ("lane_inst", K), ("lane_bytes", K), ("send_off", K + 1), ("recv_off", K + 1)):
            assert np.array_equal(got[key][b][:n], want[key][b][:n]) and (got[key][b][n:] == 77).all(), (key, b)


@pytest.mark.parametrize("name,tau", [("template_8", 0), ("template_9", 500), ("template_17", 0), ("template_17", 700)])
def test_work_order(vp, oracle_lib, name, tau):  # noqa: F811
    """More matrices than CTAs at once, of very different lengths (one empty, one invalid): the order in which they are taken
    changes no plan."""
    import torch
    cat = CATALOGS[name]()
    N = cat.topology.N
    rng = np.random.default_rng(N + tau)
    base = (rng.integers(1, 60, size=(5, N, N)) * 4096).astype(np.int64)
    for b, keep in enumerate((0.0, 0.02, 0.2, 0.05, 0.1)):
        base[b] *= rng.random((N, N)) < keep
        np.fill_diagonal(base[b], 0)
    base[4, 1, 0] = -4096
    w = WParams(granule_bytes=4096).resolved(N)
    dc = vp.load_catalog(cat.topology.blob(), cat.blob())
    p = ts._params(vp, w)
    B = vp.schedule_launch_info(dc, 1 << 14, p)["ctas"] + 3
    given = np.full(5, tau, dtype=np.int64) if tau else None
    want = oracle_lib.OracleCatalog(cat.topology.blob(), cat.blob()).schedule_batch(base, w, tau_in=given, threads=5)
    pick = np.arange(B) % 5
    got = vp.schedule_batch(dc, p, torch.from_numpy(base[pick]).cuda(), tau_ns_in=torch.from_numpy(given[pick]).cuda() if tau else None).cpu()
    for key in ts.KEYS:
        for r in range(5):
            assert (got[key][r::5] == want[key][r]).all(), (key, r)


@pytest.mark.parametrize("name,batches", [("template_3_64_50", (740, 741, 1185)), ("template_4", (740, 741, 1184, 1185, 2369)),
                                          ("template_8", (148, 149, 592, 1185)), ("template_9", (296, 593))])
def test_launch_shapes_of_node_symmetric_catalogs(vp, oracle_lib, name, batches):  # noqa: F811
    """Up to eight groups CTAs of two lanes per group are followed by CTAs of one that pack the SMs, above by CTAs of one and warps
    that emit: the last batch of a shape and the first of the next, and batches beyond one wave."""
    test_work_counters_and_batches(vp, oracle_lib, name, batches)


@pytest.mark.parametrize("name,warps", [("two_nodes_64_50", 1), ("ring_of_three", 4)])
def test_warps_per_cta_by_what_an_sm_holds(vp, oracle_lib, name, warps):  # noqa: F811
    """Six to eight matrices per SM: a warp per CTA where an SM holds as many of them, else CTAs of more warps, which share the tables (52
    KB with the 468 families of a ring of three switches); a wave holds the batch either way."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cat = CATALOGS[name]()
    dc = vp.load_catalog(cat.topology.blob(), cat.blob())
    p = ts._params(vp, WParams(granule_bytes=4096).resolved(cat.topology.N))
    for B in (6 * sms + 1, 8 * sms):
        info = vp.schedule_launch_info(dc, B, p)
        assert info["threads"] == 32 * warps and info["ctas"] == (B + warps - 1) // warps
    assert vp.schedule_launch_info(dc, 6 * sms, p)["threads"] == 64
    test_work_counters_and_batches(vp, oracle_lib, name, (7 * sms,))


def _one_rail(nodes):
    """One switch per node: every rank group keeps its four lanes, or sends one to the group `delta` further on."""
    topo = tree_topology(nodes, switches_per_node=1)
    by_key = {(r.src_group, r.dst_group): i for i, r in enumerate(topo.instances)}
    fams = [tuple(sorted(x for a in range(nodes) for x in [by_key[a, a]] * (3 if d else 4) + ([by_key[a, (a + d) % nodes]] if d else [])))
            for d in range(nodes)]
    return _assemble(topo, fams)


@pytest.mark.parametrize("nodes,rails", [(2, 2), (3, 2), (4, 2), (8, 2), (9, 2), (16, 2), (17, 2), (2, 1), (5, 1), (16, 1), (17, 1), (40, 1)])
def test_first_maximum_by_class(vp, oracle_lib, nodes, rails):  # noqa: F811
    """Step 1 class by class, a row per lane (up to sixteen groups) and in chunks, with two rails and one: shape scores that tie
    massively (every cell equal; inside the switches only; between neighbours only), a single cell, and random ones."""
    cat = node_template_catalog(tree_topology(nodes)) if rails == 2 else _one_rail(nodes)
    N = cat.topology.N
    rng = np.random.default_rng(10 * nodes + rails)
    D = (rng.integers(0, 900, size=(6, N, N)) * (rng.random((6, N, N)) < 0.3)).astype(np.int64)
    group = np.arange(N) // 4
    D[1] = 1000
    D[2] = 700 * (group[:, None] == group[None, :])
    D[3] = 500 * ((group[:, None] ^ 1) == group[None, :])
    D[4] = 0
    D[4][1, N - 2] = 77
    D *= 256
    for b in range(6):
        np.fill_diagonal(D[b], 0)
    for extra in ({}, {"k_target": N, "n_start": 3}):
        w = WParams(granule_bytes=256, k_max=12 * N, **extra).resolved(N)
        got, want, *_ = ts._both(vp, oracle_lib, cat, D, w)
        ts._assert_same(got, want)


def _reordered(nodes):
    """The node template catalog with its shapes in another order: a first row has several runs, so there are no classes."""
    cat = node_template_catalog(tree_topology(nodes))
    order = np.random.default_rng(nodes).permutation(cat.n_shapes)
    return Catalog(cat.topology, [cat.shapes[s] for s in order], [cat.buckets[s] for s in order])


def _thinned(nodes):
    """All but five or six of its shapes: the lists of second rows differ, so the classes are many."""
    cat = node_template_catalog(tree_topology(nodes))
    keep = [s for s in range(cat.n_shapes) if s % (cat.n_shapes // 5) != 7]
    return Catalog(cat.topology, [cat.shapes[s] for s in keep], [cat.buckets[s] for s in keep])


def _rails(nodes, S):
    """Three or four switches per node: every rail sends one lane to its own rail `d` nodes further on (a `d` per rail, none if 0), or
    all rails to the next rail."""
    topo = tree_topology(nodes, switches_per_node=S)
    by_key = {(r.src_group, r.dst_group, r.kind): i for i, r in enumerate(topo.instances)}

    def family(to):                                        # to(node, rail) -> the group it sends a lane to
        fam = []
        for n in range(nodes):
            for q in range(S):
                a, d = n * S + q, to(n, q)
                fam += [by_key[a, a, 0]] * (4 if d == a else 3) + ([by_key[a, d, 2]] if d != a else [])
        return tuple(sorted(fam))
    several = itertools.product(range(nodes), repeat=S) if nodes ** S < 700 else ((d,) * S for d in range(nodes))
    fams = [family(lambda n, q: (n + ds[q]) % nodes * S + q) for ds in several]
    fams += [family(lambda n, q: (n + d) % nodes * S + (q + r) % S) for r in range(1, S) for d in range(nodes)]
    return _assemble(topo, fams)


WITHOUT_CLASSES = {
    "reordered_4": lambda: _reordered(4), "reordered_8": lambda: _reordered(8), "reordered_12": lambda: _reordered(12), "reordered_17": lambda: _reordered(17),
    "thinned_4": lambda: _thinned(4), "thinned_8": lambda: _thinned(8),
    "three_rails": lambda: _rails(4, 3), "four_rails": lambda: _rails(5, 4), "three_rails_of_36_groups": lambda: _rails(12, 3),
}


@pytest.mark.parametrize("name", list(WITHOUT_CLASSES))
def test_first_maximum_without_classes(vp, oracle_lib, name):  # noqa: F811
    """Catalogs whose first maximum is not taken class by class: two rails in another order or of more classes than a lane's rows
    allow, three and four rails.  All launch shapes; scores within 32 bits and beyond."""
    cat = WITHOUT_CLASSES[name]()
    N = cat.topology.N
    dc = vp.load_catalog(cat.topology.blob(), cat.blob(), device=0)
    assert dc.node_symmetric == 1 and (dc.argmax_classes > 5 if "thinned" in name else dc.argmax_classes == 0)
    w = WParams(granule_bytes=256, k_max=8 * N).resolved(N)
    assert vp.schedule_launch_info(dc, 4, ts._params(vp, w))["kernel"] == "CTA per matrix, 16-bit credits"
    rng = np.random.default_rng(N)
    D = (rng.integers(0, 900, size=(6, N, N)) * (rng.random((6, N, N)) < 0.3)).astype(np.int64)
    D[1] = 1000
    D[2] = 0
    D[2][1, N - 2] = 77
    D[3] = rng.integers(0, 3, size=(N, N))
    D[4] *= 1 << 20                                            # scores beyond 32 bits
    D *= 256
    for b in range(6):
        np.fill_diagonal(D[b], 0)
    got, want, *_ = ts._both(vp, oracle_lib, cat, D, w)
    ts._assert_same(got, want)
    for B in (300, 700) if N <= 64 else (300,):                # the other launch shapes
        plan = vp.schedule_batch(dc, ts._params(vp, w), torch.from_numpy(np.tile(D, (-(-B // 6), 1, 1))[:B].copy()).cuda()).cpu()
        for r in range(0, B, 6):
            ts._assert_same({key: plan[key][r:r + 6] for key in ts.KEYS}, {key: want[key][:min(6, B - r)] for key in ts.KEYS})


@pytest.mark.parametrize("nodes,k_max", [(17, 120), (24, 150), (32, 300)])
def test_first_maximum_by_class_beyond_32_bits(vp, oracle_lib, nodes, k_max):  # noqa: F811
    """Matrices of 2^30 granules and more with capacities of 16 bits, in the chunks of more than sixteen groups: every cell equal (all
    scores tie; 17 nodes cross 2^30 on the way), random cells, and a cell left alone."""
    cat = node_template_catalog(tree_topology(nodes))
    N = cat.topology.N
    rng = np.random.default_rng(nodes)
    D = np.full((3, N, N), 58600 if nodes == 17 else 40000, dtype=np.int64)
    D[1] += rng.integers(0, 2800 if nodes == 17 else 20000, size=(N, N))
    D[2] = D[1] * (rng.random((N, N)) < 0.99)
    D *= 256
    for b in range(3):
        np.fill_diagonal(D[b], 0)
    assert D[0].sum() // 256 >= 1 << 30
    got, want, *_ = ts._both(vp, oracle_lib, cat, D, WParams(granule_bytes=256, k_target=4 * N, k_max=k_max).resolved(N))
    ts._assert_same(got, want)


@pytest.mark.parametrize("name", ["one_node", "two_nodes_64_50", "ring_of_three"])
@pytest.mark.parametrize("n_start,i_aa", [(1, 3), (2, 1), (3, 3), (4, 2), (5, 3), (8, 4)])
def test_starts_of_the_warp_kernel(vp, oracle_lib, name, n_start, i_aa):  # noqa: F811
    """Fewer starts than the four that fill a warp, and more: one family of a shape and several; ties between starts."""
    cat = CATALOGS[name]()
    N = cat.topology.N
    rng = np.random.default_rng(n_start)
    D = (rng.integers(0, 900, size=(6, N, N)) * (rng.random((6, N, N)) < 0.5)).astype(np.int64)
    D[1] = 1000
    D[2] = 0
    D[2][1, N - 2] = 77
    D *= 256
    for b in range(6):
        np.fill_diagonal(D[b], 0)
    got, want, *_ = ts._both(vp, oracle_lib, cat, D, WParams(granule_bytes=256, n_start=n_start, i_aa=i_aa).resolved(N))
    ts._assert_same(got, want)


def _repeated(cat, shapes):
    """The catalog with each of `shapes` followed by copies of itself: (shape, copies)."""
    order = [s for s in range(cat.n_shapes) for _ in range(1 + dict(shapes).get(s, 0))]
    return Catalog(cat.topology, [cat.shapes[s] for s in order], [cat.buckets[s] for s in order])


def _second_rows(cat):
    """Per run of shapes that share their first row: the shapes."""
    def first(shape):
        return tuple((d, c) for a, d, c in shape if a == 0)
    runs = {}
    for s, shape in enumerate(cat.shapes):
        runs.setdefault(first(shape), []).append(s)
    return list(runs.values())


@pytest.mark.parametrize("nodes,rails", [(2, 2), (4, 2), (8, 2), (9, 2), (5, 1)])
@pytest.mark.parametrize("where", ["one", "every", "ends", "long"])
def test_repeated_shapes(vp, oracle_lib, nodes, rails, where):  # noqa: F811
    """A catalog may hold a shape more than once: the first of the equal ones is chosen.  One repeated shape, all of them, the last of
    every list of second rows, and lists of more than 32 entries by repeats alone."""
    cat = node_template_catalog(tree_topology(nodes)) if rails == 2 else _one_rail(nodes)
    runs = _second_rows(cat)
    again = {"one": {cat.n_shapes // 2: 1}, "every": {s: 1 for s in range(cat.n_shapes)}, "ends": {r[-1]: 2 for r in runs},
             "long": {s: 35 for r in runs for s in r[:1]}}[where]
    cat = _repeated(cat, again)
    N = cat.topology.N
    rng = np.random.default_rng(100 * nodes + rails)
    D = (rng.integers(0, 900, size=(5, N, N)) * (rng.random((5, N, N)) < 0.3)).astype(np.int64)
    D[1] = 1000
    D[2] = 0
    D[2][1, N - 2] = 77
    D[3] = rng.integers(0, 3, size=(N, N))
    D *= 256
    for b in range(5):
        np.fill_diagonal(D[b], 0)
    got, want, *_ = ts._both(vp, oracle_lib, cat, D, WParams(granule_bytes=256, k_max=12 * N).resolved(N))
    assert (want["status"] == 0).all()
    ts._assert_same(got, want)


@pytest.mark.parametrize("granule", [256, 7392, 14336, 999983])
@pytest.mark.parametrize("nodes", [2, 4, 8, 12, 32])
def test_set_up_of_a_matrix(vp, oracle_lib, nodes, granule):  # noqa: F811
    """Entries up to the limit of 2^40 (quotients by a reciprocal; capacities in every mode), one wrong entry of each kind at the edges of
    a matrix, and demand at addresses that are multiples of eight only."""
    cat, N = node_template_catalog(tree_topology(nodes)), 8 * nodes
    rng = np.random.default_rng(nodes * 1000003 + granule)
    most = ((1 << 40) - 1) // granule
    D = np.zeros((7, N, N), dtype=np.int64)
    D[0, 0, N - 1] = D[0, N - 1, 0] = D[0, 1, 6] = most * granule
    for i, j in rng.integers(0, N, size=(9, 2)):
        if i != j:
            D[1, i, j] = int(rng.integers(1, 65536 * 3)) * granule
    D[2:] = D[1]
    D[2, N - 1, N - 2] = granule * 5 + 1
    D[3, 0, N - 1] = 1 << 40
    D[4, N - 1, N - 1] = granule
    D[5, N - 1, 0] = -granule
    D[6, N // 2, 0] = (most - 1) * granule + granule // 2
    w = WParams(granule_bytes=granule, k_max=6 * N).resolved(N)
    got, want, _, dc = ts._both(vp, oracle_lib, cat, D, w)
    ts._assert_same(got, want)
    assert want["n_steps"][:2].min() > 0 and want["status"].tolist()[2:] == [vp.ST_NOT_GRANULE, vp.ST_OVERFLOW_RISK, vp.ST_DIAG_NONZERO, vp.ST_NEGATIVE, vp.ST_NOT_GRANULE]
    flat = torch.zeros(D.size + 1, dtype=torch.int64, device="cuda")
    flat[1:] = torch.from_numpy(D).cuda().view(-1)
    ts._assert_same(vp.schedule_batch(dc, ts._params(vp, w), flat[1:].view(7, N, N)).cpu(), want)
