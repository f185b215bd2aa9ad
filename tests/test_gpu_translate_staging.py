"""The general translation with its coefficients staged in shared memory up to
the limit of 48 KB a CTA: FP64 column counts whose coefficients take 41,216
and 48,384 bytes on a cube of two wavelengths (112 translation types of one
parent, one and two lanes per output, one and two columns per thread), and
those just below and above, against single columns.  FP64 sums in another
order stay within 1e-10."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_1756_gb300 import mlfma as M  # noqa: E402


def test_staged_coefficients_up_to_the_limit():
    v, t = workloads.cube(2.0, 20)
    P = M.MlfmaPlan(v, t, 2 * np.pi, 4, 5.0, max_batch=13, precisions=(M.FP64,))
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((P.n, 13), generator=g, device="cuda", dtype=torch.float64)
    one = torch.cat([P.matvec(x[:, c:c + 1]) for c in range(13)], 1)
    for B in (2, 3, 4, 5, 6, 7, 9, 10, 11, 12, 13):
        y = P.matvec(x[:, :B].contiguous())
        assert float((y - one[:, :B]).norm() / one[:, :B].norm()) < 1e-10, B
    P.close()
