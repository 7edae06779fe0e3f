"""swkb_modes_noalloc's rounding: its split into rows and columns is no further from the exact coefficients
than rows of 2048 points summed directly."""
import math

import numpy as np
import pytest

from paper_2301_03814_gb300 import swkb

pytestmark = pytest.mark.gpu


def _field(n, n_max, seed):
    rng = np.random.default_rng(seed)
    m = np.arange(n)
    u = np.zeros(n, complex)
    for _ in range(6):
        c, width = rng.uniform(0.1, 0.9) * n, rng.uniform(0.005, 0.05) * n + 2.0
        f = rng.uniform(-0.5, 0.5) * n_max / n
        u += rng.uniform(0.3, 1.0) * np.exp(-((m - c) / width) ** 2 + 2j * math.pi * f * (m - c))
    return u


# errors measured with rows of 2048 points (n / 2048 of them) and every bin a sum of its own, over these
# very fields; their means over other fields scatter by 1 to 2 %
@pytest.mark.parametrize("n,direct", [(4096, 1.237e-16), (16384, 1.358e-16), (32768, 1.429e-16), (65536, 1.504e-16)])
def test_split_rounds_no_more_than_direct_sums(n, direct):
    torch = pytest.importorskip("torch")
    errs = []
    for i in range(24):
        n_max = int(n / 4 - 1) // (1 + i % 8)
        u = _field(n, n_max, 4000 + 500 + i)
        want = np.fft.fft(u.astype(np.clongdouble)) / n
        want = np.concatenate([want[n - n_max:], want[:n_max + 1]])
        d = torch.from_numpy(u).cuda()
        c = torch.empty(2 * n_max + 1, dtype=torch.complex128, device="cuda")
        swkb.check(swkb.swkb_modes_noalloc(d.data_ptr(), n, n_max, c.data_ptr(), torch.cuda.current_stream().cuda_stream))
        errs.append(float(np.linalg.norm((c.cpu().numpy() - want).astype(complex)) / np.linalg.norm(want.astype(complex))))
    assert math.exp(float(np.mean(np.log(errs)))) < 1.02 * direct
