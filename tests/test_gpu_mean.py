"""The mean: its tiles at every width of the rows' loads, on both sides of the
lengths at which another kind of tile takes over, and the same bits by every way
to it."""
import numpy as np
import pytest

import oracle
import synth
from _gpu_round import assert_mean_close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
ap = pytest.importorskip("paper_2108_02416_gb300")
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("K,r", [(7, 3), (9, 3), (15, 3), (24, 3)])
@pytest.mark.parametrize("d", [1, 130, 19_455, 19_457, 77_823, 77_825])
@pytest.mark.parametrize("align", [4, 2, 1])
def test_mean_of_the_kept_copies(K, r, d, align):
    a = ap.aspis_assign(K, r)
    ld = -(-d // 4) * 4 + (0 if align == 4 else 4 - align)
    gen = torch.Generator(DEV).manual_seed(K * d)
    copies = torch.randn((a.f, r, ld), device=DEV, generator=gen)
    rng = np.random.default_rng(d)
    buf = ap.RoundBuffers(a, d, DEV)
    for n in (a.f, a.f - 5, 13, 1, 0):
        sel = np.full(a.f, -1, np.int8)
        sel[np.sort(rng.permutation(a.f)[:n])] = rng.integers(0, r, n)
        buf.det.zero_()
        buf.out.fill_(7.0)
        ap.aspis_aggregate(copies, d, a, torch.from_numpy(sel).to(DEV), buf.det, buf.out, ap.MEAN)
        torch.cuda.synchronize()
        if n == 0:
            assert buf.detection().status == ap.E_EMPTY and bool((buf.out == 7.0).all())
            continue
        kept = np.nonzero(sel >= 0)[0]
        rows = torch.from_numpy(kept * r + sel[kept]).to(DEV)
        x = copies.view(-1, ld)[rows, :d].cpu().numpy()
        assert_mean_close(buf.out.cpu().numpy(), oracle.mean(x), np.abs(x.astype(np.float64)).mean(0))


@pytest.mark.parametrize("K,r,q,attack", [(15, 3, 5, "weak"), (15, 3, 3, "strong"), (9, 3, 4, "weak"), (12, 4, 5, "weak"),
                                          (11, 5, 5, "weak"), (20, 2, 6, "weak")])
@pytest.mark.parametrize("align", [4, 2, 1])
@pytest.mark.parametrize("everywhere", [True, False])
def test_every_way_to_the_mean_gives_the_same_bits(K, r, q, attack, align, everywhere):
    """The round in one call (one pass over the copies at this length, with a guessed
    selection that a distortion of one coordinate makes wrong), its four calls, the
    round without caller buffers and the one from host memory: whatever files are
    dropped, the same sums in the same order."""
    oa, a = oracle.assign(K, r), ap.aspis_assign(K, r)
    d = -(-250_000_000 // (a.f * r)) // 4 * 4 + 4
    ld = d + (0 if align == 4 else 4 - align)
    gen = torch.Generator(DEV).manual_seed(K)
    # large values that cancel among small ones: the order of summation shows
    x = torch.randn((a.f, 1, ld), device=DEV, generator=gen)
    x[0::3] *= 1e6
    x[1::3] = -x[0::3][: x[1::3].shape[0]]
    copies = x.expand(a.f, r, ld).contiguous()
    w = synth.Workload("m", K=K, r=r, d=d, q=q, attack=attack, seed=K)
    rng = np.random.default_rng(K)
    for i, s in zip(*np.nonzero(synth.corrupted_mask(w, oa.file_workers))):
        if everywhere:
            copies[int(i), int(s)] *= -2.0
        else:
            copies[int(i), int(s), int(rng.integers(d))] += 1e7
    one, four = ap.RoundBuffers(a, d, DEV), ap.RoundBuffers(a, d, DEV)
    ap.aspis_round(copies, d, a, one.file_neq, one.adj, one.det, one.sel, one.out, ap.MEAN)
    ap.aspis_check(copies, d, a, four.file_neq, four.adj)
    ap.aspis_detect(four.adj, K, four.det)
    ap.aspis_select(four.file_neq, four.det, a, four.sel)
    ap.aspis_aggregate(copies, d, a, four.sel, four.det, four.out, ap.MEAN)
    outs = [four.out.clone()]
    ap.aspis_round_static(copies, d, a, four.det, four.out, ap.MEAN)
    outs.append(four.out.clone())
    host = torch.empty(copies.shape, pin_memory=True)
    host.copy_(copies)
    host_out = torch.empty(d, pin_memory=True)
    host_det = torch.empty(ap.DETECTION_BYTES, dtype=torch.uint8, pin_memory=True)
    ap.aspis_round_host(host, copies, d, a, four.file_neq, four.adj, four.det, four.sel, four.out, host_out, host_det,
                        ap.MEAN)
    torch.cuda.synchronize()
    outs.append(host_out.to(DEV))
    if attack == "weak":
        assert one.detection().n_sel < a.f
    for out in outs:
        assert torch.equal(one.out.view(torch.int32), out.view(torch.int32))
