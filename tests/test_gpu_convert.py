"""Node bytes to bit-planes and back, and coarse-graining, at the sizes where
their kernels take another path: byte arrays off the 32-byte grid, rows that
end in padding, blocks of several words, of more than a warp of words, and
block rows that do not fill a group."""
from __future__ import annotations

import numpy as np
import pytest

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


@pytest.mark.parametrize("offset", [0, 1, 16, 32])
@pytest.mark.parametrize("W,H", [(32, 2), (64, 10), (96, 6), (128, 4), (1056, 14), (8192, 6)])
def test_bytes_and_planes(pkg, W, H, offset):
    import torch
    rng = np.random.Generator(np.random.PCG64(W + H + offset))
    s = rng.integers(0, 256, size=(H, W), dtype=np.uint8)
    raw = torch.zeros(H * W + offset, dtype=torch.uint8, device="cuda")
    t = raw[offset:].view(H, W)
    t.copy_(torch.from_numpy(s))
    with pkg.Lattice(W, H, seed=1) as lat:
        lat.set_state_tensor(t)
        words = lat.get_rows_tensor(0, H).cpu().numpy().view(np.uint32)    # [7, H, pitch]
        bits = ((words[:, :, : W // 32, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(7, H, W)
        assert np.array_equal(bits, (s[None] >> np.arange(7)[:, None, None]) & 1)
        assert not words[:, :, W // 32:].any()
        out = torch.zeros(H * W + offset, dtype=torch.uint8, device="cuda")
        lat.get_state_tensor(out=out[offset:].view(H, W))
        assert np.array_equal(out[offset:].view(H, W).cpu().numpy(), s)
        assert np.array_equal(lat.get_state(), s)


@pytest.mark.parametrize("W,H,B", [(32, 32, 32), (1056, 64, 32), (1152, 192, 96), (960, 320, 160), (2048, 1024, 1024),
                                   (3072, 1536, 1536), (640, 1280, 640), (1088, 128, 64), (4096, 4096, 4096), (8448, 128, 128),
                                   (640, 384, 128)])
@pytest.mark.parametrize("solid", [False, True])
def test_coarse_grain_blocks(pkg, oracle_mod, W, H, B, solid):
    rng = np.random.Generator(np.random.PCG64(W + H + B))
    s = rng.integers(0, 128, size=(H, W), dtype=np.uint8)
    if solid:
        s[rng.random((H, W)) < 0.3] |= 0x80
        s[:B, :B] |= 0x80                      # a block without fluid nodes
    with pkg.Lattice(W, H, seed=1) as lat:
        lat.set_state(s)
        got = lat.coarse_grain(B)
    want = oracle_mod.coarse_grain(s, B)
    assert np.array_equal(got[0], want[0])
    for g, r in zip(got[1:], want[1:]):
        np.testing.assert_allclose(g, r.astype(np.float32), rtol=1e-6, atol=1e-30)


@pytest.mark.parametrize("W,H,B", [(32, 5120, 32), (160, 9600, 32), (192, 9600, 32), (384, 12800, 64), (96, 61440, 96),
                                   (192, 122880, 96), (768, 23040, 128), (128, 19200, 128), (256, 98560, 256),
                                   (512, 97024, 256), (1024, 23040, 128)])
@pytest.mark.parametrize("solid", [False, True])
def test_coarse_grain_narrow(pkg, oracle_mod, W, H, B, solid):
    """Lattices of many short rows of blocks, on either side of the line from
    which a warp takes a block."""
    rng = np.random.Generator(np.random.PCG64(W + H + B))
    s = rng.integers(0, 128, size=(H, W), dtype=np.uint8)
    if solid:
        s[rng.random((H, W)) < 0.3] |= 0x80
        s[-B:, -B:] |= 0x80                    # a block without fluid nodes
    with pkg.Lattice(W, H, seed=1) as lat:
        lat.set_state(s)
        got = lat.coarse_grain(B)
    want = oracle_mod.coarse_grain(s, B)
    assert np.array_equal(got[0], want[0])
    for g, r in zip(got[1:], want[1:]):
        np.testing.assert_allclose(g, r.astype(np.float32), rtol=1e-6, atol=1e-30)


def test_coarse_grain_sparse_large_block(pkg, oracle_mod):
    """One block with more fluid nodes than a float counts (2^25 + 2) and few
    particles: the density is the quotient in doubles, rounded once."""
    n, mass = 8192, 1001
    s = np.zeros((n, n), dtype=np.uint8)
    s[:n // 2] = 0x80
    s[0, :2] = 0
    s[n // 2:].reshape(-1)[:mass] = 0x01
    with pkg.Lattice(n, n, seed=1) as lat:
        lat.set_state(s)
        counts, rho, ux, uy = lat.coarse_grain(n)
    fluid = 2**25 + 2
    assert counts[0, 0, 7] == fluid and counts[0, 0, 8] == mass
    assert np.float32(mass / fluid) != np.float32(mass) / np.float32(fluid)
    assert rho[0, 0] == np.float32(mass / fluid)
    want = oracle_mod.coarse_grain(s, n)
    assert ux[0, 0] == np.float32(want[2][0, 0]) and np.isclose(uy[0, 0], want[3][0, 0], rtol=1e-6)


@pytest.mark.parametrize("n,solid_rows", [(8192, 0), (8192, 4094), (4096, 0)])
def test_coarse_grain_empty_large_block(pkg, n, solid_rows):
    """A block without particles, with 2^26, a little over 2^25 and 2^24 fluid
    nodes: every field is zero."""
    with pkg.Lattice(n, n, seed=1) as lat:
        if solid_rows:
            lat.load_obstacle_shapes([(pkg.SHAPE_ROWS, 0, solid_rows, 0)])
        counts, rho, ux, uy = lat.coarse_grain(n)
    assert counts.reshape(-1).tolist() == [0] * 7 + [n * (n - solid_rows), 0]
    assert rho[0, 0] == 0.0 and ux[0, 0] == 0.0 and uy[0, 0] == 0.0
