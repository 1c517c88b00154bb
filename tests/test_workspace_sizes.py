"""Workspace sizes over brick counts (CPU: size queries of the C ABI)."""

import pytest

from paper_2009_09500_gb300 import build, vox

# dims of (64-row, 64-slice) multiples with the brick counts on both sides of every
# step of the counter replicas (512 and 32768 bricks), and beyond
BRICKS = {511: (7, 73), 512: (8, 64), 513: (9, 57), 4096: (64, 64), 32767: (1057, 31), 32768: (256, 128),
          32769: (10923, 3), 65536: (256, 256), 262144: (512, 512), 1 << 20: (1024, 1024)}


def setup_module(_):
    build.build_library()
    vox.load()


@pytest.mark.parametrize("size", ["vox_workspace_size_volume", "vox_euclid_workspace_size_volume"])
@pytest.mark.parametrize("n", [1, 5000])
def test_workspace_serves_every_smaller_volume(size, n):
    sizes = []
    for nb, (a, b) in BRICKS.items():
        dims = (256, 64 * a, 64 * b)
        assert vox.vox_scene_bricks(dims) == nb
        sizes.append(getattr(vox, size)(n, dims, 100))
    assert sizes == sorted(sizes)
    f = getattr(vox, size)
    assert f(n, (4096, 4096, 4096), 100) >= f(n, (4096, 4096, 2048), 100)


@pytest.mark.parametrize("n_scenes", [1, 300])
def test_batched_workspace_serves_every_smaller_batch(n_scenes):
    sizes = [vox.vox_workspace_size_batched_volume(5000, n_scenes, nb, 100) for nb in BRICKS]
    assert sizes == sorted(sizes)
