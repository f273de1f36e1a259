"""Helpers for the GPU parity tests: run one round through the C ABI and run
the oracle on the same bytes."""
import numpy as np

import bench


def as_u32(t):
    return t.detach().cpu().numpy().view(np.uint32)


def spoil(u, rng):
    """Columns of u (uint32 [f, d]) that no tile settles: groups of 32 with 1, 2, 5,
    6, 7, 12, 17 and 32 of them, of every kind (equal values, a few, a bin or an
    8-bit counter too full, NaNs, infinities, extreme keys), and single ones at both
    ends."""
    f, d = u.shape
    i = np.arange(f)
    far = rng.standard_normal(f).astype(np.float32) + np.where(i % 10 < 3, 100, 0).astype(np.float32)
    kinds = [np.zeros(f), np.full(f, 0x3F800000),
             np.where(i % 2, 0x3F800000, 0xBF800000), np.where(i % 3, 0, 0x80000000),
             np.where(i % 5, 0, rng.integers(0, 1 << 32, f)), i % 7,
             np.where(i == f // 2, 0x7FC00001, u[:, 0]), np.where(i % 2, 0x7F800000, 0xFF800000),
             np.where(i % 2, 0xFFFFFFFF, 0x7FFFFFFF), rng.integers(0, 1 << 32, f),
             far.view(np.uint32),
             np.where(i % 4, 0xFFFFFFFF, u[:, 0]), np.where(i % 4, 0x7F7FFFFF, 0xFF7FFFFF)]
    spots = {0, d - 1}
    for g, many in enumerate([1, 2, 5, 6, 7, 12, 17, 32]):
        if 32 * g + 32 <= d:
            spots.update(32 * g + rng.permutation(32)[:many])
    spots.update(rng.integers(0, d, d // 300))
    for k, c in enumerate(sorted(spots)):
        u[:, c] = kinds[(k * 5 + k // len(kinds)) % len(kinds)]


def takes_one_pass(ap, torch, copies_dev, d, a, mode=0):
    """Whether aspis_round reads the copies in one pass: by the kernels it enqueues."""
    buf = ap.RoundBuffers(a, d, copies_dev.device)
    stream = torch.cuda.Stream()

    def call():
        ap.aspis_round(copies_dev, d, a, buf.file_neq, buf.adj, buf.det, buf.sel, buf.out, mode, stream)

    with torch.cuda.stream(stream):
        call()
    stream.synchronize()
    return bench.captured_kernels(torch, stream, call) >= bench.ONE_PASS_KERNELS


def gpu_round(ap, torch, copies_dev, d, a, mode=0, stream=None):
    """copies_dev: CUDA float32 [f, r, ld] (any storage offset)."""
    buf = ap.RoundBuffers(a, d, copies_dev.device)
    ap.aspis_round(copies_dev, d, a, buf.file_neq, buf.adj, buf.det, buf.sel, buf.out, mode,
                   stream)
    torch.cuda.synchronize()
    return buf


def assert_round_matches(ap, buf, want, mode=0, check_out=True):
    det = buf.detection()
    assert det.status == ap.OK, ap.status_str(det.status)
    assert np.array_equal(as_u32(buf.file_neq), want.file_neq), "file_neq"
    assert np.array_equal(as_u32(buf.adj), want.adj), "adjacency"
    got = (det.omega, det.n_max_cliques, det.clique_mask, bool(det.success))
    assert got == (want.det.omega, want.det.n_max, want.det.clique, want.det.success), "clique"
    assert np.array_equal(buf.sel.cpu().numpy(), want.sel), "sel"
    assert det.n_sel == want.n_sel, "n_sel"
    if check_out:
        out = buf.out.cpu().numpy()
        if mode == 0:
            assert np.array_equal(out.view(np.uint32), want.out.view(np.uint32)), \
                f"median mismatch at {np.nonzero(out.view(np.uint32) != want.out.view(np.uint32))[0][:10]}"
        else:
            assert_mean_close(out, want.out, None)


def assert_mean_close(got, want, scale):
    """|gpu - oracle| <= 1e-6 * max(|oracle|, mean|x|) + 1e-30 (mean mode)."""
    ref = np.abs(want.astype(np.float64))
    if scale is not None:
        ref = np.maximum(ref, scale)
    err = np.abs(got.astype(np.float64) - want.astype(np.float64))
    bad = err > 1e-6 * ref + 1e-30
    assert not bad.any(), f"mean mismatch at {np.nonzero(bad)[0][:10]}"
