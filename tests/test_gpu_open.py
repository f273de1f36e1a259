"""Coordinates that the tile kernel cannot settle and leaves open: equal values,
crowded bins, NaNs and infinities, few or many of them in a group of 32, with as
many rows as fill a warp's share or leave a remainder."""
import statistics

import numpy as np
import pytest

import oracle
from _gpu_round import as_u32, spoil

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
ap = pytest.importorskip("paper_2108_02416_gb300")
DEV = torch.device("cuda:0")


# the files' number, the rows' alignment and d decide which tiles leave them open, and
# who settles them: the tile's own block (one tile per SM) or the kernel after it
@pytest.mark.parametrize("K,r", [(8, 3), (15, 3), (12, 4), (16, 3), (18, 3), (12, 6), (20, 3), (21, 3)])
@pytest.mark.parametrize("d,odd", [(300, 0), (19_600, 0), (19_600, 2), (19_601, 1)])
def test_open_coordinates(K, r, d, odd):
    oa, a = oracle.assign(K, r), ap.aspis_assign(K, r)
    rng = np.random.default_rng(K * d)
    f, ld = oa.f, d + odd
    host = np.zeros((f, r, ld), np.float32)
    host[:] = rng.standard_normal((f, 1, ld), dtype=np.float32)
    plane = host[:, 0].view(np.uint32).copy()
    spoil(plane[:, :d], rng)
    host[:] = plane.view(np.float32)[:, None, :]
    dev = torch.from_numpy(host).to(DEV)
    for n in (f, f - 1, f // 32 * 32, f // 32 * 32 + 1, 33, 2, 1):
        if not 0 < n <= f:
            continue
        sel = np.full(f, -1, np.int8)
        sel[np.sort(rng.permutation(f)[:n])] = rng.integers(0, r, n)
        buf = ap.RoundBuffers(a, d, DEV)
        buf.det.zero_()
        ap.aspis_aggregate(dev, d, a, torch.from_numpy(sel).to(DEV), buf.det, buf.out)
        torch.cuda.synchronize()
        want = oracle.aggregate(host, sel, 0, 0, d)
        bad = np.nonzero(as_u32(buf.out) != want.view(np.uint32))[0]
        assert bad.size == 0, (n, bad[:8])
        assert buf.detection().median_exact > 0


@pytest.mark.parametrize("K,r,d", [(9, 3, 524_288), (15, 3, 262_144), (18, 3, 131_072)])
def test_a_tenth_of_equal_values(K, r, d):
    """Units that are off make a tenth of the coordinates equal in all files: the
    aggregation takes 1.5 to 3 times as long as without (57 and 18 times with four
    passes over the rows in global memory); 6 leaves room for a busy machine."""
    a = ap.aspis_assign(K, r)
    gen = torch.Generator(DEV).manual_seed(1)
    copies = torch.randn((a.f, 1, d), device=DEV, generator=gen).expand(a.f, r, d).contiguous()
    sel = torch.zeros(a.f, dtype=torch.int8, device=DEV)
    buf = ap.RoundBuffers(a, d, DEV)
    buf.det.zero_()

    def timed():
        times = []
        for _ in range(9):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            ap.aspis_aggregate(copies, d, a, sel, buf.det, buf.out)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return statistics.median(times[2:])

    plain = timed()
    copies[:, :, torch.rand(d, device=DEV, generator=gen) < 0.1] = 0.0
    tied = timed()
    assert buf.detection().median_exact > d // 20
    assert tied < 6 * plain, (plain, tied)
