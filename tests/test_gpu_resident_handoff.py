"""The shared-memory resident kernel's hand-off of edge rows: one SM alone,
strips of exactly two rows, several quads per thread, wide rows, and step counts
of either parity, bit-exact with the oracle."""
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


@pytest.mark.parametrize("W,H", [(32, 2), (256, 256), (128, 640), (160, 320), (96, 642), (2048, 42), (512, 304),
                                 (512, 306), (512, 512), (1056, 1024), (256, 48), (4128, 300), (4096, 2048), (24576, 4), (12320, 310), (16384, 64)])
@pytest.mark.parametrize("p", [0.0, 0.03])
def test_handoff(pkg, oracle_mod, W, H, p):
    seed = 5 * W + H
    s0 = workloads.bernoulli_lattice(W, H, 0.3, seed, workloads.channel_walls(W, H) if p and H > 2 else None)
    with pkg.Lattice(W, H, seed=seed, forcing_p=p) as lat:
        assert lat.step_kernel == 4 and lat.temporal_block in (1, 2, 4)      # the automatic choice
        lat.set_state(s0)
        for n in (1, 2, 7, 4, 13):
            lat.step(n)
        assert lat.t == 27
        got = lat.get_state()
    want, _ = oracle_mod.run(s0, seed, 0, 27, p)
    assert np.array_equal(got, want), f"{int((got != want).sum())} nodes differ"
