"""The brick binning at its edges (GPU): segments whose lengths lie around the units
that a lane walks, volumes on both sides of the unit rule and longer than 2^17 along
one axis, few and many bricks (counter replicas); piece counts against the oracle's
voxels and the documented brick shape, whole volumes against the oracle."""

import numpy as np
import pytest

from gpu_util import brick_pieces_expected, bricked_from_row_major, get_oracle, run_gpu
from paper_2009_09500_gb300 import batching, vox, workloads

pytestmark = pytest.mark.gpu


def _segs(rng, dims, n):
    """Uniform segments, and axis-near ones whose length is 255..257, 511..513 or the
    volume's whole extent."""
    segs = workloads.uniform_segments(rng, n, dims)
    for i in range(0, n, 2):
        a = int(rng.integers(0, 3))
        length = min(int(rng.choice([0, 1, 255, 256, 257, 511, 512, 513, 1 << 21])), dims[a] - 1)
        segs[i, a] = rng.integers(0, dims[a] - length)
        segs[i, a + 3] = segs[i, a] + length
        if rng.random() < 0.5:
            segs[i] = np.concatenate([segs[i, 3:], segs[i, :3]])
    return segs


@pytest.mark.parametrize("dims", [(512, 512, 64), (544, 96, 512), (1024, 1024, 64), (262144, 64, 33), (32, 40000, 64)])
def test_binning_edges(dims):
    rng = np.random.default_rng(sum(dims))
    segs = _segs(rng, dims, 403)
    O = get_oracle()
    r = run_gpu(segs, dims, vox.OUT_BITMASK | vox.OUT_FRESH, pieces="plan")
    assert r["status"] == 0
    assert r["planned"][1] == brick_pieces_expected(O, segs, dims)
    assert np.array_equal(r["mask"], O.bitmask(segs, dims))


def test_binning_batched_few_and_many_bricks():
    """One small scene (replicated counters) and the same scene beside larger ones."""
    rng = np.random.default_rng(8)
    O = get_oracle()
    small = workloads.Workload("s", _segs(rng, (64, 64, 64), 5000), (64, 64, 64))
    large = workloads.Workload("l", _segs(rng, (1024, 1024, 512), 300), (1024, 1024, 512))
    for scenes in ([small], [large, small, large, small]):
        b = batching.make_batch(scenes, vox.OUT_BITMASK | vox.OUT_FRESH)
        assert b.pieces == sum(brick_pieces_expected(O, s.segs, s.dims) for s in scenes)
        b.run()
        assert int(b.status.item()) == 0
        for m, s in zip(b.masks, scenes):
            assert np.array_equal(m.cpu().numpy().view(np.uint32), O.bitmask(s.segs, s.dims))


@pytest.mark.parametrize("dims", [(64, 64, 64), (128, 128, 96), (160, 70, 130), (256, 256, 100)])
@pytest.mark.parametrize("flags", [vox.OUT_BITMASK, vox.OUT_BITMASK | vox.OUT_FRESH, vox.OUT_BITMASK | vox.OUT_BRICKED])
def test_bricks_walked_in_parts(dims, flags):
    """Many pieces in few bricks: several CTAs walk a brick, whose bits are OR-ed into a
    volume that is kept, cleared first, or brick-major; over stale bits."""
    rng = np.random.default_rng(sum(dims))
    segs = workloads.uniform_segments(rng, 9000, dims)
    bricked = bool(flags & vox.OUT_BRICKED)
    words = vox.vox_mask_words_bricked(dims) if bricked else vox.vox_mask_words(dims)
    init = rng.integers(0, 2**32, size=words, dtype=np.uint64).astype(np.uint32)
    r = run_gpu(segs, dims, flags, mask_init=init, pieces="plan", mask_words=words)
    want = get_oracle().bitmask(segs, dims)
    if bricked:
        want = bricked_from_row_major(want, dims)
    elif not flags & vox.OUT_FRESH:
        want = want | init
    assert r["status"] == 0
    assert np.array_equal(r["mask"], want)
