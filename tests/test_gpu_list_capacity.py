"""Lists whose buffer is larger than the total (GPU): the same list, in the same time."""

import numpy as np
import pytest
import torch

from gpu_util import get_oracle
from paper_2009_09500_gb300 import vox, workloads

pytestmark = pytest.mark.gpu
UNBOUNDED = 2**63 - 1


def _scan(w):
    segs = vox.segments_tensor(w.segs)
    ws = torch.full((vox.vox_workspace_size(w.n),), 0xA5, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    vox.vox_count(segs, w.dims, ws, st)
    return segs, ws, st


@pytest.mark.parametrize("bits", [32, 64])
def test_large_capacities_give_the_same_list(bits):
    """More than one chunk per resident warp (5e7 voxels), and far less than one; several
    lists of one scan."""
    O = get_oracle()
    rng = np.random.default_rng(bits)
    for n, top in ((98_000, 1024), (300, 200)):
        w = workloads.Workload("m", workloads._segments_from_major(rng, rng.integers(0, top, n), 1024), (1024,) * 3)
        want = O.list32(w.segs) if bits == 32 else O.list64(w.segs)
        V = len(want)
        segs, ws, st = _scan(w)
        out = torch.empty(V + 64, dtype=torch.int32 if bits == 32 else torch.int64, device="cuda")
        flag = vox.OUT_LIST32 if bits == 32 else vox.OUT_LIST64
        for capacity in (V, 3 * V, UNBOUNDED, V):
            out.fill_(-1)
            vox.vox_generate_from_scan(segs, w.dims, ws, st, out, None, flag, capacity=capacity)
            got = out.cpu().numpy().view(want.dtype)
            assert int(st.item()) == 0
            assert np.array_equal(got[:V], want) and (out[V:] == -1).all(), capacity


def test_both_list_types_of_one_scan_on_two_streams():
    rng = np.random.default_rng(3)
    w = workloads.Workload("m", workloads._segments_from_major(rng, rng.integers(0, 1024, 80_000), 1024), (1024,) * 3)
    O = get_oracle()
    segs, ws, st = _scan(w)
    l32 = torch.empty(O.total(w.segs), dtype=torch.int32, device="cuda")
    l64 = torch.empty(len(l32), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for out, flag in ((l32, vox.OUT_LIST32), (l64, vox.OUT_LIST64)):
        vox.vox_generate_from_scan(segs, w.dims, ws, st, out, None, flag, torch.cuda.Stream())
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert np.array_equal(l32.cpu().numpy().view(np.uint32), O.list32(w.segs))
    assert np.array_equal(l64.cpu().numpy().view(np.uint64), O.list64(w.segs))


def test_time_does_not_depend_on_the_capacity():
    """2e8 64-bit voxels: told of a capacity 3 and 16 times the total, the list takes as
    long as with the total (chunks cut from the capacity took 1.3 and 6 times as long)."""
    w = workloads.sweep_giga(200_000_000, n=1024, seed=2, edge=1 << 21)
    segs, ws, st = _scan(w)
    V = 200_000_000
    out = torch.empty(V, dtype=torch.int64, device="cuda")

    def us(capacity):
        ts = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            vox.vox_generate_from_scan(segs, w.dims, ws, st, out, None, vox.OUT_LIST64, capacity=capacity)
            b.record()
            torch.cuda.synchronize()
            ts.append(1e3 * a.elapsed_time(b))
        return sorted(ts)[3]

    us(V)
    base = us(V)
    for k in (3, 16):
        assert us(k * V) < 1.15 * base
    assert int(st.item()) == 0
