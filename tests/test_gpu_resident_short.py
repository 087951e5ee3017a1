"""Calls of as many steps as the resident kernel takes between exchanges of
edge rows (or fewer): the strips then run without waiting for one another."""
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


@pytest.mark.parametrize("p", [0.0, 0.02])
@pytest.mark.parametrize("W,H,interval,n", [(512, 304, 4, 4), (512, 1218, 4, 4), (96, 5000, 4, 4), (2048, 1024, 2, 2),
                                            (4096, 612, 2, 2), (4128, 1000, 2, 2)])
def test_calls_without_an_exchange(pkg, oracle_mod, W, H, interval, n, p):
    """interval 4: the automatic choice; 2: kernel 4 with temporal block 2."""
    seed = 3 * W + H
    s0 = workloads.bernoulli_lattice(W, H, 0.3, seed, workloads.channel_walls(W, H) if p else None)
    with pkg.Lattice(W, H, seed=seed, forcing_p=p) as lat:
        if interval == 2:
            lat.set_step_kernel(4)
            lat.set_temporal_block(2)
        lat.set_state(s0)
        assert lat.step_kernel == 4 and lat.temporal_block == interval
        for _ in range(5):
            lat.step(n)
        lat.step(n + 1)
        lat.step(n)
        got = lat.get_state()
        t = lat.t
    assert t == 7 * n + 1
    want, _ = oracle_mod.run(s0, seed, 0, t, p)
    assert np.array_equal(got, want), f"{int((got != want).sum())} nodes differ"


@pytest.mark.parametrize("W,H,p", [(32384, 4, 0.0), (24608, 6, 0.02), (16384, 32, 0.0), (32768, 2, 0.02), (1024, 8, 0.0)])
def test_short_calls_of_flat_lattices(pkg, oracle_mod, W, H, p):
    """Calls on either side of the number of steps from which the automatic
    choice keeps a flat lattice in shared memory."""
    seed = W + H
    s0 = workloads.bernoulli_lattice(W, H, 0.3, seed, workloads.channel_walls(W, H) if p and H > 2 else None)
    with pkg.Lattice(W, H, seed=seed, forcing_p=p) as lat:
        lat.set_state(s0)
        for n in range(3, 13):
            lat.step(n)
        got = lat.get_state()
    want, _ = oracle_mod.run(s0, seed, 0, sum(range(3, 13)), p)
    assert np.array_equal(got, want), f"{int((got != want).sum())} nodes differ"
