"""swkb_modes_noalloc over the splits of its DFT (one pass, and pass 1 of 2 to 64
rows with 4 or 8 columns per block), bins at the edges of the pairs, against numpy."""
import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fft", [64, 128, 256, 1024, 4096, 8192, 32768, 65536])
@pytest.mark.parametrize("part", [0.001, 0.01, 0.06, 0.2, 0.5])
def test_noalloc_modes_over_the_splits(n_fft, part):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n_fft)
    u = rng.standard_normal(n_fft) + 1j * rng.standard_normal(n_fft)
    u_dev = torch.from_numpy(u).cuda()
    top = max(1, min(int(n_fft * part), n_fft // 2 - 2))
    for n_max in (top, top + 1):
        c = torch.full((2 * n_max + 3,), 7.0, dtype=torch.complex128, device="cuda")
        assert swkb.swkb_modes_noalloc(u_dev.data_ptr(), n_fft, n_max, c.data_ptr()) == swkb.SWKB_OK
        got = c.cpu().numpy()
        want = np.fft.fft(u)[np.arange(-n_max, n_max + 1) % n_fft] / n_fft
        # sums of N1 and N2 terms: rms error about eps sqrt(N1 + N2) of the rms
        assert np.max(np.abs(got[:-2] - want)) <= 1e-12 * np.max(np.abs(want))
        assert np.all(got[-2:] == 7.0)   # nothing beyond the kept modes
