"""The mean: its tiles at every width of the rows' loads, on both sides of the
lengths at which another kind of tile takes over."""
import numpy as np
import pytest

import oracle
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
