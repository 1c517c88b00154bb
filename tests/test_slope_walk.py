"""The brick path's slopes (a host model) over their whole range of steps, and volumes
on both sides of their limit of 37,837 voxels an edge (GPU, against the oracle)."""

import numpy as np
import pytest

from paper_2009_09500_gb300 import batching, vox, workloads
from test_entry_division import estimate_and_correct

EDGE = 37837                  # longest edge with slopes
N_MAX = 65533                 # int(sqrt(3) (EDGE - 1)): the Euclidean variant's longest segment
ONE = np.uint64(1 << 40)


# ------------------------------------------------------------------ host model
def _slopes(A, N):
    """ceil(A 2^40 / N) by the kernel's two divisions of 20 bits each; 1 - 2^-40 for A = N."""
    q1, r1 = estimate_and_correct(A << 20, N)
    q2, r2 = estimate_and_correct(r1 << 20, N)
    S = (q1 << 20) + q2 + (r2 > 0)
    return np.where(A == N, (1 << 40) - 1, S).astype(np.uint64)


def _check_walk(N, A, k0, steps=64):
    """The entry at step k0 by one multiplication, then `steps` steps by 32-bit carries,
    against the offsets of Eq. (3)."""
    S = _slopes(A, N)
    exact = -((-A.astype(object) << 40) // N)  # ceil, in Python integers
    assert np.array_equal(S.astype(object), np.where(A == N, (1 << 40) - 1, exact))
    P = k0.astype(np.uint64) * S + (ONE >> np.uint64(1))
    q = (P >> np.uint64(40)).astype(np.int64)
    f = (((P >> np.uint64(8)) & np.uint64(0xffffffff)).astype(np.int64) + 1) & 0xffffffff
    s = (S >> np.uint64(8)).astype(np.int64)
    s += (s != 0xffffffff) & ((S & np.uint64(0xff)) != 0)
    for i in range(steps):
        k = k0 + i
        ok = k <= N
        assert np.array_equal(q[ok], ((2 * k * A + N) // (2 * N))[ok])
        f = f + s
        q = q + (f >> 32)
        f &= 0xffffffff


def test_short_segments_in_full():
    N = np.repeat(np.arange(1, 65), np.arange(1, 65) + 1)
    A = np.concatenate([np.arange(n + 1) for n in range(1, 65)])
    _check_walk(N, A, np.zeros_like(N))


@pytest.mark.parametrize("n_lo", [1, 4096, 32768, N_MAX - 64])
def test_random_and_extreme_segments(n_lo):
    rng = np.random.default_rng(n_lo)
    m = 60000
    N = np.where(rng.random(m) < 0.5, rng.integers(n_lo, N_MAX + 1, m), N_MAX - rng.integers(0, 64, m))
    A = rng.integers(0, N + 1)
    pick = rng.random(m)
    A = np.where(pick < 0.2, N - rng.integers(0, 3, m).clip(max=N), A)
    A = np.where((pick >= 0.2) & (pick < 0.3), rng.integers(0, 3, m).clip(max=N), A)
    A = np.where((pick >= 0.3) & (pick < 0.5), N // rng.integers(2, 9, m), A)  # ties
    k0 = np.where(rng.random(m) < 0.3, (N - 63).clip(min=0), rng.integers(0, N + 1))
    _check_walk(N, A, k0)


# ------------------------------------------------------------------------- GPU
def _segments(rng, dims, n):
    """Uniform segments, and as many from end to end of the longest axis, both ways."""
    segs = workloads.uniform_segments(rng, n, dims)
    a = int(np.argmax(dims))
    segs[::2, a], segs[::2, a + 3] = 0, dims[a] - 1
    segs[::4] = np.concatenate([segs[::4, 3:], segs[::4, :3]], axis=1)
    return segs


DIMS = [(64, EDGE, 33), (64, EDGE + 1, 33), (37824, 40, 64), (32, 96, EDGE), (4128, 70, 65), (19968, 33, 40)]


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [vox.OUT_BITMASK, vox.OUT_BITMASK | vox.OUT_FRESH])
@pytest.mark.parametrize("dims", DIMS)
def test_long_edges(dims, flags):
    from gpu_util import get_oracle, run_gpu

    segs = _segments(np.random.default_rng(sum(dims)), dims, 300)
    r = run_gpu(segs, dims, flags, pieces="plan")
    assert r["status"] == 0 and r["planned"][1] > 300
    assert np.array_equal(r["mask"], get_oracle().bitmask(segs, dims))


@pytest.mark.gpu
@pytest.mark.parametrize("dims", DIMS)
def test_long_edges_euclid(dims):
    import torch

    from gpu_util import get_oracle

    segs_np = _segments(np.random.default_rng(sum(dims)), dims, 300)
    segs, n = vox.segments_tensor(segs_np), len(segs_np)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(vox.vox_euclid_workspace_size_volume(n, dims, 0), dtype=torch.uint8, device="cuda")
    pieces = vox.vox_euclid_plan(segs, dims, ws, st, with_pieces=True)[2]
    ws = torch.empty(vox.vox_euclid_workspace_size_volume(n, dims, pieces), dtype=torch.uint8, device="cuda")
    mask = torch.full((vox.vox_mask_words(dims),), -1, dtype=torch.int32, device="cuda")
    vox.vox_euclid_generate(segs, dims, ws, st, None, mask, vox.OUT_BITMASK | vox.OUT_FRESH)
    assert int(st.item()) == 0 and pieces > 300
    assert np.array_equal(mask.cpu().numpy().view(np.uint32), get_oracle().euclid_bitmask(segs_np, dims))


@pytest.mark.gpu
def test_long_edges_batched():
    """Scenes with and without slopes side by side."""
    from gpu_util import get_oracle

    rng = np.random.default_rng(1)
    scenes = [workloads.Workload("s", _segments(rng, d, 200), d) for d in DIMS + [(64, 64, 64)]]
    b = batching.make_batch(scenes, vox.OUT_BITMASK | vox.OUT_FRESH)
    b.run()
    assert int(b.status.item()) == 0 and b.total_bricks > 0
    for m, s in zip(b.masks, scenes):
        assert np.array_equal(m.cpu().numpy().view(np.uint32), get_oracle().bitmask(s.segs, s.dims))
