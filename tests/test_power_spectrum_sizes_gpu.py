"""The snapshot spectrum at the sizes where its passes change shape: transforms that share a block or take
one alone, blocks of 64 to 512 threads, strips that end inside q_x = 0 .. Lx/2; against numpy."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import capi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Lz", [(4, 2), (2, 4), (64, 64), (512, 256), (1024, 2048), (2048, 1024), (4096, 32), (32, 4096),
                                   (8192, 512), (256, 8192)])
def test_against_numpy(Lx, Lz):
    phi = np.random.default_rng(Lx + Lz).standard_normal((Lz, Lx))
    dev = torch.from_numpy(phi).cuda()
    out = torch.full_like(dev, float("nan"))
    torch.cuda.synchronize()
    capi.lb_power_spectrum(dev.data_ptr(), Lx, Lz, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    want = np.abs(np.fft.fft2(phi)) ** 2 / (Lx * Lz)
    # both transforms round log2(n) times (up to 21): a few 1e-15 of the largest bin, bound as for the oracle
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=1e-12 * want.max())
