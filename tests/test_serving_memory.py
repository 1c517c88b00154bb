"""What admission reserves for a request covers what the launcher allocates (CPU: size
queries of the C ABI)."""

import numpy as np
import pytest

from paper_2009_09500_gb300 import build, vox
from paper_2009_09500_gb300.serving import ServeRequest


def setup_module(_):
    build.build_library()
    vox.load()


def _allocated(reqs):
    """The launcher's workspace, volumes and segments of one batch."""
    n = sum(r.n for r in reqs)
    bricks = [vox.vox_scene_bricks(r.dims) for r in reqs]
    total = sum(bricks) if n and all(bricks) else 0
    ws = vox.vox_workspace_size_batched_volume(n, len(reqs), total, sum(r.piece_capacity for r in reqs))
    return ws + sum(4 * vox.vox_mask_words(r.dims) for r in reqs) + 24 * max(n, 1)


@pytest.mark.parametrize("sizes", [(1,), (5, 1000), (1000, 100_000)])
def test_reserved_bytes_cover_the_allocations(sizes):
    rng = np.random.default_rng(len(sizes))
    edges = [1, 31, 32, 33, 64, 96, 128, 160, 256, 512, 1024]
    for _ in range(200):
        step = 32 if rng.random() < 0.7 else 1
        reqs = []
        for i in range(int(rng.integers(1, 65))):
            w, h, d = (int(rng.choice(edges)) for _ in range(3))
            reqs.append(ServeRequest(rid=i, arrival_s=0.0, n=int(rng.integers(0, sizes[-1] + 1)),
                                     dims=(max(step, w // step * step), h, d)))
        assert _allocated(reqs) <= sum(r.device_bytes for r in reqs)


def test_many_bricks():
    """Batches on both sides of the steps of the counter replicas."""
    for dims, k in [((256, 64, 64), 512), ((256, 64, 64), 513), ((1024, 1024, 1024), 32), ((1024, 1024, 1024), 33),
                    ((2048, 2048, 2048), 1), ((4096, 4096, 4096), 1)]:
        reqs = [ServeRequest(rid=i, arrival_s=0.0, n=1, dims=dims) for i in range(k)]
        assert _allocated(reqs) <= sum(r.device_bytes for r in reqs)


def test_brick_counts():
    rng = np.random.default_rng(0)
    for _ in range(500):
        dims = (int(rng.integers(1, 70)) * int(rng.choice([1, 32])), int(rng.integers(1, 3000)), int(rng.integers(1, 3000)))
        assert ServeRequest(rid=0, arrival_s=0.0, n=1, dims=dims).bricks == vox.vox_scene_bricks(dims)
