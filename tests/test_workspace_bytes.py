"""gs_workspace_bytes never falls as a problem grows, so one workspace serves every smaller problem
(host only, no GPU needed)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def size():
    import torch  # noqa: F401  (loads the CUDA runtime the library links against)
    from paper_2603_09621_gb300 import build, gs
    build.build()
    lib = gs.load()

    def f(n, capacity, nx, nz=8, brick=(8, 8, 8), det=1):
        g, c = gs.Grid(nx, 8, nz).c(), gs.Config(brick=brick, deterministic=det).c()
        return lib.gs_workspace_bytes(n, capacity, ctypes.byref(g), ctypes.byref(c))
    return f


# bricks along x at the edges of the digit widths: one pass up to 512, two up to 262,144, three beyond
BRICKS = [1, 2, 3, 255, 256, 257, 511, 512, 513, 1024, 1025, 16_384, 16_385, 131_072, 131_073, 262_144, 262_145,
          1 << 20]
GAUSS = [0, 1, 63, 64, 65, 255, 257, 38_911, 38_912, 38_913, 45_000, 155_000, 156_000, 399_999, 400_000, 4_000_000]


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("capacity", [0, 20_000, 400_000, 30_000_000])
def test_workspace_grows_with_the_cloud(size, capacity, det):
    for nb in (1, 512, 513, 131_072):
        got = [size(n, capacity, 8 * nb, det=det) for n in GAUSS]
        assert got == sorted(got) and got[0] > 0, nb


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("capacity", [0, 20_000, 400_000, 30_000_000])
def test_workspace_grows_with_the_bricks(size, capacity, det):
    for n in (1, 38_912, 500_000):
        got = [size(n, capacity, 8 * nb, det=det) for nb in BRICKS]
        assert got == sorted(got) and got[0] > 0, n
        # the same voxels in fewer, larger bricks
        assert size(n, capacity, 8 * 512, brick=(8, 8, 8), det=det) <= size(n, capacity, 8 * 512, brick=(8, 8, 4),
                                                                              det=det)


def test_workspace_grows_with_the_capacity(size):
    for n in (1, 38_912, 500_000):
        for nb in (512, 513, 262_145):
            got = [size(n, cap, 8 * nb) for cap in (0, 1, 2047, 2048, 2049, 8192, 8193, 1_000_000, 2**31 - 4096)]
            assert got == sorted(got) and got[0] > 0
