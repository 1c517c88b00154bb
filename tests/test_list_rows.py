"""The list kernel's fixed-point slopes (a host model) and its rows, windows and
chunks at their edges (GPU, whole lists against the oracle)."""

import numpy as np
import pytest

from paper_2009_09500_gb300 import vox, workloads


# ------------------------------------------------------------------ host model
def _fixed_point(S0, d, N, k, F, bits):
    """Coordinate of voxel k as the kernel computes it: the integer part of
    X0 + k T in `bits`-bit words with F fraction bits (Python integers)."""
    A = abs(d)
    S = 1 << F if A == N else -((-A << F) // N) if N else 0
    X0 = (S0 << F) + (1 << (F - 1)) - (1 if d < 0 else 0)
    return ((X0 + k * (S if d >= 0 else -S)) & ((1 << bits) - 1)) >> F


def _exact(S0, d, N, k):
    q = (2 * k * abs(d) + N) // (2 * N) if N else 0
    return S0 + q if d >= 0 else S0 - q


@pytest.mark.parametrize("F,bits,n_max", [(22, 32, 1023), (43, 64, (1 << 21) - 1)])
def test_fixed_point_coordinates_are_exact(F, bits, n_max):
    """The bound (N + 1) 2^-F <= 1 / 2N holds for the longest segment, and the
    model equals Eq. (3) on ties, extremes and random segments, both signs."""
    assert (n_max + 1) * 2 * n_max <= 1 << F
    rng = np.random.default_rng(F)
    cases = [(n_max, a, k) for a in (0, 1, n_max // 2, n_max - 1, n_max) for k in (0, 1, n_max // 2, n_max - 1, n_max)]
    for _ in range(20000):
        N = int(rng.integers(0, n_max + 1)) if rng.random() < 0.5 else n_max - int(rng.integers(0, 50))
        cases.append((N, int(rng.integers(0, N + 1)), int(rng.integers(0, N + 1))))
    for N in range(1, 40):
        cases += [(N, A, k) for A in range(N + 1) for k in range(N + 1)]
    for N, A, k in cases:
        for d in (A, -A):
            S0 = 0 if d >= 0 else A  # the segment lies at the low edge: one step off would wrap
            assert _fixed_point(S0, d, N, k, F, bits) == _exact(S0, d, N, k), (N, d, k)
            S0 = n_max - A if d >= 0 else n_max  # ... and at the high edge
            assert _fixed_point(S0, d, N, k, F, bits) == _exact(S0, d, N, k), (N, d, k)


# ------------------------------------------------------------------------- GPU
def _lengths(name, rng):
    return {
        "ones": np.ones(20000, np.int64),                               # 32 segments in 32 voxels
        "short": rng.integers(1, 7, 20000),                             # several starts per lane
        "row-1": np.full(900, 127), "row": np.full(900, 128), "row+1": np.full(900, 129),
        "half-row": np.full(2000, 64), "lane-ends": 4 * rng.integers(1, 40, 3000),
        "mixed": np.where(rng.random(4000) < 0.1, rng.integers(500, 1000, 4000), rng.integers(1, 5, 4000)),
        "one": np.array([1]), "one-row": np.array([128]), "chunk": np.array([256, 1, 255, 1000]),
        "window": np.concatenate([np.full(31, 4), [900], np.full(33, 3), [700], np.full(64, 1), [33]]),
    }[name]


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("name", ["ones", "short", "row-1", "row", "row+1", "half-row", "lane-ends", "mixed", "one",
                                  "one-row", "chunk", "window"])
def test_list_rows(name, bits):
    from gpu_util import assert_list_equal, get_oracle, run_gpu

    rng = np.random.default_rng(5)
    segs = workloads._segments_from_major(rng, np.asarray(_lengths(name, rng), np.int64) - 1, 1024)
    O = get_oracle()
    want = O.list32(segs) if bits == 32 else O.list64(segs)
    # a capacity far above the total gives the grid more rounds and the warps smaller chunks
    for capacity in (None, len(want) + 31_000_000) if name == "mixed" else (None,):
        r = run_gpu(segs, (1024,) * 3, vox.OUT_LIST32 if bits == 32 else vox.OUT_LIST64, capacity=capacity)
        assert r["status"] == 0
        assert_list_equal(r["list_full"], want, len(want))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 4095, 4096, 4097])  # one CTA's count + scan, and the tiled one
def test_small_scan(n):
    """Counts, offsets and list on both sides of the line between the two scans, with a
    status word and a workspace that hold anything before the call; an endpoint outside."""
    import torch

    from gpu_util import get_oracle

    rng = np.random.default_rng(n)
    dims = (300, 200, 100)
    segs = workloads.uniform_segments(rng, n, dims)
    O = get_oracle()
    want, off = O.list32(segs), np.concatenate([[0], np.cumsum(O.count(segs).astype(np.int64))])
    d = torch.from_numpy(segs).cuda()
    ws = torch.full((vox.vox_workspace_size(n),), 0xA5, dtype=torch.uint8, device="cuda")
    status = torch.full((1,), 4, dtype=torch.int32, device="cuda")
    counts = torch.empty(n, dtype=torch.int32, device="cuda")
    offsets = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    vox.vox_count(d, dims, ws, status, counts, offsets)
    assert int(status.item()) == 0
    assert np.array_equal(offsets.cpu().numpy(), off) and np.array_equal(counts.cpu().numpy(), np.diff(off))
    lst = torch.zeros(len(want), dtype=torch.int32, device="cuda")
    ws.fill_(0x5A)
    status.fill_(4)
    vox.vox_generate(d, dims, ws, status, lst)
    assert int(status.item()) == 0 and np.array_equal(lst.cpu().numpy().view(np.uint32), want)
    d[n - 1, 5] = 100
    lst.zero_()
    vox.vox_generate(d, dims, ws, status, lst)
    assert int(status.item()) == vox.ERR_OUT_OF_BOUNDS and int(lst.abs().sum()) == 0
