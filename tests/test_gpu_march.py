"""Register marching (passes of 2 or 3 steps with the intermediate time levels
in registers): bit-exact with the oracle on every way columns are dealt to
lanes and rows to bands, and the automatic choice of it with the direct step
kernel."""
from __future__ import annotations

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2428_gb300 import build as cuda_build
    cuda_build.build()
    import paper_1208_2428_gb300 as p
    p.load()
    return p


# Whole rows in a warp (1, 2, 3, 16, 32 quads; partial last quads) and chains
# of columns cut every 30 or 28 lanes (33 and more quads; last quads of 1, 2,
# 3 and 4 words); heights of one band, of several, and with a short last band.
SIZES = [(32, 8), (96, 14), (256, 26), (352, 10), (2048, 14), (3968, 8), (4096, 38), (4128, 10), (4160, 14),
         (4192, 26), (4224, 8), (8192, 22), (8224, 14), (29984, 10)]


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("W,H", SIZES)
@pytest.mark.parametrize("variant", ["periodic", "walls_rare", "points_dense", "fhp1", "fhp3"])
def test_march_matches_oracle(pkg, oracle_mod, W, H, k, variant):
    seed = 31 * W + H + k
    rng = np.random.Generator(np.random.PCG64(seed))
    solid, p, rules = {"periodic": (None, 0.0, 2), "walls_rare": (workloads.channel_walls(W, H), 0.02, 2),
                       "points_dense": (workloads.random_points(W, H, 0.05, rng), 0.3, 2),
                       "fhp1": (workloads.channel_walls(W, H), 0.0, 1),
                       "fhp3": (None, 0.01, 3)}[variant]
    s0 = workloads.bernoulli_lattice(W, H, 0.35, seed, solid)
    with pkg.Lattice(W, H, seed=seed, forcing_p=p) as lat:
        lat.set_rules(rules)
        lat.set_state(s0)
        lat.set_time(2**32 - 5)          # the steps pass a carry of the time counter
        lat.step_march(k, k)             # one pass: no waits
        lat.step_march(k, 6 * k)         # passes that wait for one another
        got = lat.get_state()
        assert lat.t == 2**32 - 5 + 7 * k
    want, _ = oracle_mod.run(s0, seed, 2**32 - 5, 7 * k, p, rules=rules)
    assert np.array_equal(got, want), f"{int((got != want).sum())} nodes differ"


def test_march_every_candidate_forced_and_full(pkg, oracle_mod):
    W, H = 4160, 12
    for fill in (0x7F, 0x20, 0xFF):
        s0 = np.full((H, W), fill, dtype=np.uint8)
        with pkg.Lattice(W, H, seed=9, forcing_p=1.0) as lat:
            lat.set_state(s0)
            lat.step_march(2, 8)
            got = lat.get_state()
        want, _ = oracle_mod.run(s0, 9, 0, 8, 1.0)
        assert np.array_equal(got, want)


@pytest.mark.parametrize("W,H,p,block", [(8192, 2560, 0.0, 2), (16384, 4096, 0.0, 3), (16384, 2560, 5e-4, 2),
                                         (12032, 3400, 1e-3, 2)])
def test_automatic_choice_equals_direct_kernel(pkg, W, H, p, block):
    import torch
    got = []
    for kernel in (0, 1):
        with pkg.Lattice(W, H, seed=5, forcing_p=p, step_kernel=kernel) as lat:
            lat.load_obstacle_shapes(workloads.cylinder_shapes(W, H))
            lat.init_random(0.3)
            if kernel == 0:
                assert lat.temporal_block_kernel == 3 and lat.temporal_block == block
            lat.step(17)
            got.append(lat.get_state_tensor())
            lat.synchronize()
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("W,H,p,rules", [(32, 400_000, 0.02, 2), (96, 400_000, 0.02, 1), (384, 140_000, 0.02, 2),
                                         (1152, 45_000, 0.0, 3), (2176, 15_000, 0.02, 2), (4192, 8_000, 0.02, 2),
                                         (2560, 22_000, 0.02, 2), (3040, 20_000, 0.02, 3), (1024, 60_000, 0.02, 2)])
def test_single_steps_of_large_lattices_equal_direct_kernel(pkg, W, H, p, rules):
    """Lattices beyond L2 whose rows are narrow or leave lanes empty (ragged ones
    among them), on either side of the rule's lines: single steps and calls of
    several against the direct kernel."""
    import torch
    got = []
    for kernel in (0, 1):
        with pkg.Lattice(W, H, seed=6, forcing_p=p, step_kernel=kernel) as lat:
            lat.set_rules(rules)
            lat.load_obstacle_shapes(workloads.cylinder_shapes(W, H))
            lat.init_random(0.3)
            for n in (1, 1, 4):
                lat.step(n)
            got.append(lat.get_state_tensor())
            lat.synchronize()
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("W,p", [(7_200_000, 0.0), (7_200_032, 0.0), (9_600_000, 0.0), (9_600_000, 5e-4)])
def test_rows_too_wide_to_march(pkg, W, p):
    """Rows of more columns than the warps of one resident wave hold (7.0 million
    nodes for passes of 3 steps, 9.3 million for 2 on 152 SMs): the automatic
    choice steps them with a kernel that can."""
    import torch
    H, got = 8, []
    for kernel in (0, 1):
        with pkg.Lattice(W, H, seed=5, forcing_p=p, step_kernel=kernel) as lat:
            lat.load_obstacle_shapes([(pkg.SHAPE_ROWS, 0, 1, 0), (pkg.SHAPE_DISC, W // 2, 4, 2)])
            lat.init_random(0.3)
            lat.step(7)
            got.append(lat.get_state_tensor())
            lat.synchronize()
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("W,H,p,block", [(32, 600_000, 0.0, 3), (32, 700_000, 0.0, 0), (128, 400_000, 5e-4, 2),
                                         (128, 480_000, 5e-4, 0), (96, 500_000, 0.0, 3), (160, 240_000, 0.0, 2)])
def test_automatic_choice_for_narrow_rows(pkg, W, H, p, block):
    """Rows of one quad on either side of the lines of the automatic choice (0:
    they do not march), and rows of two quads, against the direct kernel."""
    import torch
    got = []
    for kernel in (0, 1):
        with pkg.Lattice(W, H, seed=5, forcing_p=p, step_kernel=kernel) as lat:
            lat.load_obstacle_shapes(workloads.cylinder_shapes(W, H))
            lat.init_random(0.3)
            if kernel == 0:
                assert (lat.temporal_block_kernel, lat.temporal_block) == ((3, block) if block else (0, 1))
            lat.step(11)
            got.append(lat.get_state_tensor())
            lat.synchronize()
    assert torch.equal(got[0], got[1])


def test_march_refusals(pkg):
    with pkg.Lattice(64, 6, seed=1) as lat:
        lat.step_march(2, 0)
        for k, n in [(1, 2), (4, 4), (2, 3), (3, 6), (2, -2)]:   # (k = 3 needs 8 rows)
            with pytest.raises(pkg.FhpError):
                lat.step_march(k, n)
        assert lat.t == 0


def test_batch_members_march(pkg, oracle_mod):
    """A batch with automatic settings marches the members that can (any row
    width, rare forcing) and steps the others (two rows, dense forcing) singly:
    every member equals its oracle run over calls of 1 to 67 steps and with
    step budgets, with and without forced members (passes of 2 and of 3)."""
    rng = np.random.Generator(np.random.PCG64(3))
    sizes = [(32, 8), (96, 40), (128, 128), (320, 200), (1056, 66), (2048, 30), (4128, 26), (8224, 14), (256, 2), (640, 4)]
    for forced in (False, True):
        jobs = [workloads.Lattice(f"m{i}", W, H, float(rng.uniform(0.1, 0.5)), 700 + i,
                                  {1: 0.01, 4: 0.001, 3: 0.3}.get(i, 0.0) if forced else 0.0, 0,
                                  obstacle="points" if i % 2 else "none", point_frac=0.02)
                for i, (W, H) in enumerate(sizes)]
        states = [j.initial_state() for j in jobs]
        with pkg.Batch(sum(pkg.Batch.lattice_bytes(j.W, j.H) for j in jobs) + (64 << 20)) as b:
            slots = []
            for j, s0 in zip(jobs, states):
                k = b.add(j.W, j.H, j.seed, j.p)
                b.set_state(k, s0)
                b.set_time(k, 2**32 - 9)
                slots.append(k)
            b.set_rules(slots[2], 1)
            b.set_steps_left(slots[5], 11)
            for n in (2, 3, 4, 5, 67, 1):
                b.step(n)
            b.synchronize()
            for i, (j, s0, k) in enumerate(zip(jobs, states, slots)):
                n = 11 if i == 5 else 82
                want, _ = oracle_mod.run(s0, j.seed, 2**32 - 9, n, j.p, rules=1 if i == 2 else 2)
                assert b.time(k) == 2**32 - 9 + n
                assert np.array_equal(b.get_state(k), want), (j.W, j.H, forced)


def test_batch_of_more_members_than_a_launch_holds(pkg, oracle_mod):
    """300 members: more than one group of 256; a wide one among them."""
    jobs = [(64, 16, 900 + i, 0.3) for i in range(299)] + [(8192, 64, 1300, 0.2)]
    with pkg.Batch(sum(pkg.Batch.lattice_bytes(w, h) for w, h, *_ in jobs) + (32 << 20)) as b:
        slots = []
        for w, h, seed, rho in jobs:
            k = b.add(w, h, seed, 0.0)
            b.init_random(k, rho)
            slots.append(k)
        b.step(6)
        for i in (0, 255, 256, 298, 299):
            w, h, seed, rho = jobs[i]
            want, _ = oracle_mod.run(oracle_mod.init_random(w, h, seed, rho), seed, 0, 6, 0.0)
            assert np.array_equal(b.get_state(slots[i]), want), i


def _mixed(kind):
    """Members beside which an untuned batch marches, or does not."""
    big = [(2048, 2048, 0.0)] * 10
    return {"all": [(512, 384, 0.0)] * 6,
            "one dense": [(512, 384, 0.0)] * 6 + [(256, 256, 0.02)],
            "many plain, one flat": big + [(2048, 4, 0.0)],
            "many plain, one dense": [(4096, 4096, 0.0)] * 9 + [(512, 512, 0.02)],
            "forced and dense": [(1024, 512, 1e-3)] * 8 + [(512, 512, 0.02)],
            "one column": [(64, 65536, 1e-3)] * 10,
            "two groups": [(64, 32, 1e-3)] * 300,
            "forced, many": [(128, 64, 1e-3)] * 150}[kind]


@pytest.mark.parametrize("kind,marches", [("all", {2: 1, 3: 1, 5: 1, 66: 1}), ("one dense", {2: 0, 3: 0, 5: 0, 66: 0}),
                                          ("many plain, one flat", {2: 1, 3: 1, 5: 1, 66: 1}),
                                          ("many plain, one dense", {2: 0, 3: 0, 5: 1, 66: 1}),
                                          ("forced and dense", {2: 0, 3: 0, 5: 0, 66: 0}),
                                          ("one column", {2: 0, 3: 0, 5: 0, 66: 0}),
                                          ("two groups", {4: 1, 3: 0, 5: 0, 66: 0}),
                                          ("forced, many", {2: 1, 3: 0, 5: 0, 66: 1})])
def test_untuned_batches_march_where_it_pays(pkg, kind, marches):
    """The route of every length of call (by its launches: single steps take one
    a step) and the members' states against a batch of single steps."""
    members = _mixed(kind)
    arena = sum(pkg.Batch.lattice_bytes(w, h) for w, h, _ in members) + (32 << 20)
    with pkg.Batch(arena) as a, pkg.Batch(arena) as b:
        b.set_step_kernel(1)
        b.set_temporal_block(1)
        for x in (a, b):
            for i, (w, h, p) in enumerate(members):
                assert x.add(w, h, 50 + i, p) == i
                x.init_random(i, 0.3)
        for n, want in marches.items():
            before = a.kernel_launches, b.kernel_launches
            a.step(n)
            b.step(n)
            single = b.kernel_launches - before[1]
            assert single == n
            rest = any(h < 6 or p >= 0.01 for _, h, p in members)      # (steps of their own)
            got = a.kernel_launches - before[0]
            assert (got != n) == bool(want) if not rest or not want else got > n, (n, got)
        a.synchronize()
        b.synchronize()
        for i in sorted({0, 1, len(members) // 2, len(members) - 2, len(members) - 1}):
            assert a.time(i) == b.time(i) == sum(marches)
            assert np.array_equal(a.get_state(i), b.get_state(i)), members[i]


def test_captured_batch_step_replays(pkg):
    """A captured call of a batch that has marched before, replayed: its passes
    wait for one another at every replay, and calls between and after the replays
    are not disturbed."""
    import torch
    stream = torch.cuda.Stream()
    members = [(2048, 1536), (512, 300), (4160, 512), (96, 2000)]
    arena = sum(pkg.Batch.lattice_bytes(w, h) for w, h in members) + (32 << 20)
    with pkg.Batch(arena, stream=stream) as a, pkg.Batch(arena, stream=stream) as b:
        b.set_step_kernel(1)
        b.set_temporal_block(1)
        for x in (a, b):
            for i, (w, h) in enumerate(members):
                x.add(w, h, 70 + i, 0.0)
                x.init_random(i, 0.3)
            x.step(18)                     # (an even number of passes, as below)
            x.synchronize()
        graph = torch.cuda.CUDAGraph()
        launches = a.kernel_launches
        with torch.cuda.graph(graph, stream=stream):
            a.step(12)                     # the graph: steps 18 .. 29, from and to the same buffers
        assert a.kernel_launches - launches == 1
        with torch.cuda.stream(stream):
            for _ in range(3):
                graph.replay()
                a.step(6)                  # steps 30 .. 35, 36 .. 41, 42 .. 47
            graph.replay()
        for start in (30, 36, 42, None):
            for i in range(len(members)):
                b.set_time(i, 18)
            b.step(12)
            if start is not None:
                for i in range(len(members)):
                    b.set_time(i, start)
                b.step(6)
        a.synchronize()
        b.synchronize()
        for i in range(len(members)):
            assert np.array_equal(a.get_state(i), b.get_state(i)), members[i]
